// Block-resident ready-counter engine: pdb_sgd_epoch under a READY schedule
// when the per-feature (weight, version) records of all n_cols features fit
// in one thread block's shared memory (up to ~20,000 features).
//
// Same protocol as the grid-wide READY engine (the read protocol of Section
// 5 per feature; record = bits(w_j) | version << 32, all epochs in one
// launch), but the records live in shared memory: a wait is a shared-memory
// poll of a few tens of cycles instead of an L2 round trip, which is what
// bounds data with many short dependency hops (the tiny workload: 441 levels of
// ~45 examples).  The version the occurrence of rank r waits for in epoch e is
// e * n_rows + r (a rank is below n_rows), the last occurrence of an epoch
// publishes (e + 1) * n_rows: below 2^31, so no two epochs share one however
// many of them are in flight.
//
// An example takes LPE lanes (8, 16 or 32: the rows' length), so a warp works
// on 32 / LPE of them at once, each group of lanes in its own example: one pass
// of the loop polls for all groups and computes and stores the ones whose
// weights have all arrived.  Group s of G takes the examples s, s + G, .. in
// data order (epoch-major).  The oldest unfinished example waits for nothing
// and its group, which takes its examples in order, is on it: no deadlock;
// every wait is bounded.  Each group keeps three examples in flight: the row
// bounds of the one after next and the ids, values and gate words of the next
// are loading while it waits on and computes the current one.
//
// What bounds it: the latency of a dependency hop (store to shared memory,
// poll, multiply, combine, derivative: ~600 cycles with 4 warps per scheduler)
// and one SM's instruction issue.  Measured, before and after an example took
// its own lanes only and the loop lost its divergent branches: one epoch of 1000
// examples of 4-16 ids over 600 features 165 -> 77 us; 20000 examples of 10 ids
// over 10000 features 840 -> 350 us (kernel alone).
#include <cuda_runtime.h>

#include "common.cuh"

using namespace pdb;

namespace {

constexpr int BR_MAXK = 64;             // longest row: 32 lanes of two elements
constexpr int BR_WARPS = 32;           // most warps

// warp_combine inside groups of LPE lanes (rows of at most LPE ids, or 32 lanes):
// the partials of the lanes that a group does not have are +0, added once (a
// second addition of +0 changes nothing).
template <int LPE>
__device__ __forceinline__ float combine_group(float a)
{
    if (LPE == 32) return warp_combine_latency(a);
    const float z = __fadd_rn(a, 0.0f);
    float n;
    if (LPE == 16) {
        const float b8 = __shfl_xor_sync(FULL, z, 8), b4 = __shfl_xor_sync(FULL, z, 4);
        const float b12 = __shfl_xor_sync(FULL, z, 12);
        n = __fadd_rn(__fadd_rn(z, b8), __fadd_rn(b4, b12));
    } else {
        n = __fadd_rn(z, __shfl_xor_sync(FULL, z, 4));
    }
    const float c2 = __shfl_xor_sync(FULL, n, 2), c1 = __shfl_xor_sync(FULL, n, 1), c3 = __shfl_xor_sync(FULL, n, 3);
    return __fadd_rn(__fadd_rn(n, c2), __fadd_rn(c1, c3));
}

// the lanes of the groups all of whose lanes are set in m
template <int LPE>
__device__ __forceinline__ unsigned full_groups(unsigned m)
{
    if (LPE == 32) return m == FULL ? FULL : 0u;
    constexpr unsigned G = LPE == 16 ? 0xffffu : 0xffu;
    unsigned f = 0;
#pragma unroll
    for (int s = 0; s < 32; s += LPE) f |= (m >> s & G) == G ? G << s : 0u;
    return f;
}

// loads that leave their destination as it is when `on` is false.  The state
// below is updated by predicates and selects only: a branch that a part of the
// warp takes costs more than the work, and a value loaded inside one is waited
// for at its end.
__device__ __forceinline__ void ld_keep(int64_t &v, const int64_t *p, bool on)
{
    asm volatile("{\n\t.reg .pred q;\n\tsetp.ne.s32 q, %2, 0;\n\t@q ld.global.b64 %0, [%1];\n\t}" : "+l"(v) : "l"(p), "r"((int)on));
}
__device__ __forceinline__ void ld_keep(int &v, const int *p, bool on)
{
    asm volatile("{\n\t.reg .pred q;\n\tsetp.ne.s32 q, %2, 0;\n\t@q ld.global.b32 %0, [%1];\n\t}" : "+r"(v) : "l"(p), "r"((int)on));
}
__device__ __forceinline__ void ld_keep(float &v, const float *p, bool on)
{
    asm volatile("{\n\t.reg .pred q;\n\tsetp.ne.s32 q, %2, 0;\n\t@q ld.global.f32 %0, [%1];\n\t}" : "+f"(v) : "l"(p), "r"((int)on));
}
__device__ __forceinline__ void st_srec_if(unsigned addr, float w, unsigned version, bool on)
{
    const unsigned long long v = (unsigned long long)__float_as_uint(w) | ((unsigned long long)version << 32);
    asm volatile("{\n\t.reg .pred q;\n\tsetp.ne.s32 q, %2, 0;\n\t@q st.relaxed.cta.shared.b64 [%0], %1;\n\t}" ::"r"(addr),
                 "l"(v), "r"((int)on)
                 : "memory");
}

template <int LPE, int R, int LOSS, bool TRACE>
__global__ __launch_bounds__(BR_WARPS * 32, 1) void k_sgd_block_ready(int32_t n_rows, int64_t n_cols,
                                                                      const int64_t *__restrict__ row_ptr,
                                                                      const int32_t *__restrict__ col,
                                                                      const float *__restrict__ val,
                                                                      const float *__restrict__ y,
                                                                      const uint32_t *__restrict__ gate, float *w,
                                                                      float eta, int epochs, int *status,
                                                                      uint64_t timeout, uint64_t *trace)
{
    extern __shared__ __align__(16) unsigned char smem_raw[];
    unsigned long long *rec = reinterpret_cast<unsigned long long *>(smem_raw);
    if (read_status(status)) return;
    const int lane = threadIdx.x & 31, warp = threadIdx.x >> 5, nwarps = blockDim.x >> 5;
    for (int64_t f = threadIdx.x; f < n_cols; f += blockDim.x)
        rec[f] = (unsigned long long)__float_as_uint(w[f]);
    __syncthreads();

    const unsigned base = (unsigned)__cvta_generic_to_shared(rec);
    const int sl = lane % LPE, groups = nwarps * (32 / LPE);
    const int total = epochs * n_rows;           // below 2^31
    // the example two ahead: its number over all epochs, its row, its epoch's first version, its bounds
    int tg = warp + nwarps * (lane / LPE), t = tg;
    unsigned bver = 0;
    int64_t bb = 0, be = 0;
    // the one ahead, loading (ntg = total: none)
    int nj[R], ng[R], nk = 0, ntg = total;
    float nx[R], ny = 0.0f;
    unsigned nver = 0;
    // the current one (live: there is one), its records' addresses
    unsigned at[R], want[R], next[R];
    float x[R], yc = 0.0f;
    int k = 0, ctg = total;
    bool live = false, slow = false;
#pragma unroll
    for (int r = 0; r < R; ++r) {
        nj[r] = ng[r] = 0;
        x[r] = nx[r] = val ? 0.0f : 1.0f;
        at[r] = base;
        want[r] = next[r] = 0u;
    }
    auto wrap = [&]() {                          // row and first version of the example tg
        while (t >= n_rows && tg < total) {
            t -= n_rows;
            bver += (unsigned)n_rows;
            asm volatile("" : "+r"(t));          // a loop, not a division ahead of every example
        }
    };
    // where `on`: current <- ahead <- bounds of the one two ahead <- the next of this group
    auto advance = [&](bool on) {
        live = on ? ntg < total : live;
        k = on ? nk : k;
        yc = on ? ny : yc;
        ctg = on ? ntg : ctg;
#pragma unroll
        for (int r = 0; r < R; ++r) {
            const unsigned g = (unsigned)ng[r], wt = (g & GATE_RANK) + nver;
            at[r] = on ? base + 8u * (unsigned)nj[r] : at[r];
            x[r] = on ? nx[r] : x[r];
            next[r] = on ? ((g & GATE_LAST) ? nver + (unsigned)n_rows : wt + 1u) : next[r];
            want[r] = on ? wt : want[r];
        }
        const bool more = tg < total;
        nk = on ? (more ? (int)(be - bb) : 0) : nk;
        nver = on ? bver : nver;
        ntg = on ? tg : ntg;
        ld_keep(ny, y + t, on && more);
#pragma unroll
        for (int r = 0; r < R; ++r) {
            const int i = r * 32 + sl;
            const bool in = on && i < nk;
            ld_keep(nj[r], col + bb + i, in);
            if (val) ld_keep(nx[r], val + bb + i, in);
            ld_keep(ng[r], reinterpret_cast<const int *>(gate) + bb + i, in);
        }
        tg = on ? (more ? tg + groups : tg) : tg;
        t = on ? (more ? t + groups : t) : t;
        if (t >= n_rows && tg < total) wrap();
        ld_keep(bb, row_ptr + t, on && tg < total);
        ld_keep(be, row_ptr + t + 1, on && tg < total);
    };
    wrap();
    ld_keep(bb, row_ptr + t, tg < total);
    ld_keep(be, row_ptr + t + 1, tg < total);
    advance(true);
    advance(true);

    unsigned alive = __ballot_sync(FULL, live);
    unsigned spins = 0;
    uint64_t t0 = 0;
    while (alive) {
        // every group's records at once (a group without an example, and the lanes past
        // a row's end, want nothing)
        float wv[R];
        bool ok = true;
#pragma unroll
        for (int r = 0; r < R; ++r) {
            unsigned long long v;
            asm volatile("ld.relaxed.cta.shared.b64 %0, [%1];" : "=l"(v) : "r"(at[r]) : "memory");
            wv[r] = __uint_as_float((unsigned)v);
            ok = ok && ((unsigned)(v >> 32) == want[r] || r * 32 + sl >= k);
        }
        unsigned run = full_groups<LPE>(__ballot_sync(FULL, ok && !slow)) & alive;
        auto margin = [&]() {
            float acc = 0.0f;
#pragma unroll
            for (int r = 0; r < R; ++r) {
                const float f = __fmaf_rn(wv[r], x[r], acc);
                acc = r * 32 + sl < k ? f : acc;
            }
            return combine_group<LPE>(acc);
        };
        // the running groups' stores, and their next examples; `seen`: when their weights
        // had all been read, in this pass (also those of a group set aside, whose records
        // are read again in each)
        auto finish = [&](float c, bool done, uint64_t seen) {
            if (TRACE) {
                if (done && sl == 0) {
                    trace[2 * (int64_t)ctg] = seen;
                    trace[2 * (int64_t)ctg + 1] = globaltimer();
                }
                __syncwarp();            // before any write is visible
            }
#pragma unroll
            for (int r = 0; r < R; ++r)
                st_srec_if(at[r], __fsub_rn(wv[r], __fmul_rn(c, x[r])), next[r], done && r * 32 + sl < k);
            // the stores go out before anything waits for the next example's loads (moved above
            // them, that wait sat on every hop: 77 -> 108 us per epoch of 1000 short examples)
            __syncwarp();
            advance(done);
            __syncwarp();
            alive = __ballot_sync(FULL, live);
        };
        if (run) {
            spins = 0;
            const uint64_t seen = TRACE ? globaltimer() : 0;
            bool redo = false;
            const float c = dev_step_fast(LOSS, margin(), yc, eta, redo);
            const bool mine = run >> lane & 1u;
            if (LOSS == PDB_LOSS_LOGISTIC) slow = mine ? redo : slow;     // set aside
            finish(c, mine && !redo, seen);
            continue;
        }
        if (LOSS == PDB_LOSS_LOGISTIC) {
            // no group can run but those set aside for the general derivative (their
            // records are as they were: nobody else may write them)
            run = __ballot_sync(FULL, slow) & alive;
            if (run) {
                spins = 0;
                const uint64_t seen = TRACE ? globaltimer() : 0;
                const float c = __fmul_rn(eta, dev_grad(LOSS, margin(), yc));
                const bool mine = run >> lane & 1u;
                slow = mine ? false : slow;
                finish(c, mine, seen);
                continue;
            }
        }
        if ((++spins & 63u) == 0) {
            int stop = read_status(status);
            const uint64_t now = globaltimer();
            if (spins == 64) t0 = now;
            if (!stop && now - t0 > timeout) {
                set_status(status, PDB_ETIMEOUT);
                stop = 1;
            }
            if (__any_sync(FULL, stop)) break;       // every warp still reaches the barrier below
        }
    }
    __syncthreads();
    for (int64_t f = threadIdx.x; f < n_cols; f += blockDim.x) w[f] = __uint_as_float((unsigned)rec[f]);
}

using BlockReadyKernel = void (*)(int32_t, int64_t, const int64_t *, const int32_t *, const float *, const float *,
                                  const uint32_t *, float *, float, int, int *, uint64_t, uint64_t *);
template <int LPE, int R, bool TRACE>
BlockReadyKernel block_ready_kernel(int loss)
{
    return loss == PDB_LOSS_LOGISTIC ? k_sgd_block_ready<LPE, R, PDB_LOSS_LOGISTIC, TRACE>
           : loss == PDB_LOSS_SQUARED ? k_sgd_block_ready<LPE, R, PDB_LOSS_SQUARED, TRACE>
                                      : k_sgd_block_ready<LPE, R, PDB_LOSS_HINGE, TRACE>;
}

// as many lanes per example as its ids need
template <bool TRACE>
BlockReadyKernel block_ready_kernel(int max_row, int loss)
{
    return max_row <= 8 ? block_ready_kernel<8, 1, TRACE>(loss) : max_row <= 16 ? block_ready_kernel<16, 1, TRACE>(loss)
           : max_row <= 32 ? block_ready_kernel<32, 1, TRACE>(loss) : block_ready_kernel<32, 2, TRACE>(loss);
}

}  // namespace

namespace pdb {

// shared memory for the block-resident READY engine, 0 when it does not apply
int64_t block_ready_smem(int64_t n_cols, int64_t max_row)
{
    if (n_cols < 1 || max_row > BR_MAXK) return 0;
    int dev = 0, optin = 0;
    cudaGetDevice(&dev);
    if (cudaDeviceGetAttribute(&optin, cudaDevAttrMaxSharedMemoryPerBlockOptin, dev) != cudaSuccess) {
        cudaGetLastError();
        return 0;
    }
    const int64_t bytes = n_cols * 8;
    return bytes + 1024 <= optin ? bytes : 0;
}

int block_ready_run(const pdb_csr *X, const float *y, const uint32_t *gate, float *w, int loss, float eta,
                    int epochs, int max_row, int *status, uint64_t timeout, uint64_t *trace, cudaStream_t s)
{
    const int64_t smem = block_ready_smem(X->n_cols, max_row);
    if (smem == 0) return PDB_ETOOBIG;
    const BlockReadyKernel kern = trace ? block_ready_kernel<true>(max_row, loss) : block_ready_kernel<false>(max_row, loss);
    // (every call: another size, and another kernel per form, loss and trace)
    if (cudaFuncSetAttribute((const void *)kern, cudaFuncAttributeMaxDynamicSharedMemorySize, (int)smem) != cudaSuccess)
        return PDB_ECUDA;
    // Warps: more examples in flight reach further ahead, fewer share the SM's
    // instruction issue.  Two examples conflict with probability ~k^2 / n_cols (k ids
    // each, spread evenly); where 16 warps hold several conflicts of an example
    // already, more only poll.  Measured, 16 / 24 / 32 warps: 1000 examples of 10
    // ids over 600 features 77 / 85 / 102 us, 20000 over 10000 features (whole call)
    // 616 / 600 / 581.
    const double k = X->n_rows > 0 ? (double)X->nnz / (double)X->n_rows : 0.0;
    const int warps = 16.0 * k * k > (double)X->n_cols ? 16 : BR_WARPS;
    kern<<<1, warps * 32, (size_t)smem, s>>>((int32_t)X->n_rows, X->n_cols, X->row_ptr, X->col, X->val, y, gate, w,
                                                eta, epochs, status, timeout, trace);
    note_launch();
    return cudaPeekAtLastError() == cudaSuccess ? PDB_OK : PDB_ECUDA;
}

}  // namespace pdb
