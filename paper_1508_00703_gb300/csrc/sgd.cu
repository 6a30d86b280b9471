// Update engines: pdb_sgd_epoch's level-synchronous and ready-counter
// dataflow engines and its dispatch to the others (window.cu, blockready.cu,
// chain.cu, resident.cu); the host side of pdb_ssp_epoch (kernels in
// ssp.cu); pdb_bsp_epoch (the BSP mini-batch comparison).
//
// In the two engines here one warp runs one example (one transaction,
// Definition 3): the lanes load the example's ids and values with coalesced
// loads, gather w through L2, form the margin with per-lane fused
// multiply-adds and a xor-shuffle combine, compute the scalar eta*g, and
// scatter w_j -= eta*g*x_j.  No atomics touch w: the schedule guarantees
// that no other example holds any of these features at the same time.
#include <cuda.h>
#include <cuda_runtime.h>

#include <algorithm>
#include <new>
#include <mutex>

#include "common.cuh"

using namespace pdb;

namespace {



// ---------------------------------------------------------------- one example, no waits
// Used by the level-synchronous engine: the level schedule already keeps
// every example of a level disjoint from the others (Theorem 3).  Element i
// of the row lives in lane i mod 32, register i / 32; each lane accumulates
// its elements in increasing i with fused multiply-adds, then the lanes
// combine pairwise (the fixed order both sides of the parity check use).
template <int R>
__device__ __forceinline__ void sgd_example(int t, const int64_t *__restrict__ row_ptr, const int32_t *__restrict__ col,
                                            const float *__restrict__ val, const float *__restrict__ y, float *w,
                                            int loss, float eta, uint64_t *trace, int64_t idx)
{
    const int lane = threadIdx.x & 31;
    const int64_t b = row_ptr[t];
    const int k = (int)(row_ptr[t + 1] - b);
    const float yt = y[t];
    float acc = 0.0f;
    if (k <= 32 * R) {
        int j[R];
        float x[R], wv[R];
#pragma unroll
        for (int r = 0; r < R; ++r) {
            int i = r * 32 + lane;
            j[r] = i < k ? col[b + i] : 0;
            x[r] = i < k ? (val ? val[b + i] : 1.0f) : 0.0f;
        }
#pragma unroll
        for (int r = 0; r < R; ++r)
            if (r * 32 + lane < k) wv[r] = __ldcg(w + j[r]);
#pragma unroll
        for (int r = 0; r < R; ++r)
            if (r * 32 + lane < k) acc = __fmaf_rn(wv[r], x[r], acc);
        const float m = warp_combine(acc);       // every lane's loads have returned
        trace_mark(trace, idx, 0);
        const float c = __fmul_rn(eta, dev_grad(loss, m, yt));
        trace_mark(trace, idx, 1);   // before any write is visible
#pragma unroll
        for (int r = 0; r < R; ++r)
            if (r * 32 + lane < k) __stcg(w + j[r], __fsub_rn(wv[r], __fmul_rn(c, x[r])));
    } else {
        for (int i = lane; i < k; i += 32) acc = __fmaf_rn(__ldcg(w + col[b + i]), val ? val[b + i] : 1.0f, acc);
        const float m = warp_combine(acc);
        trace_mark(trace, idx, 0);
        const float c = __fmul_rn(eta, dev_grad(loss, m, yt));
        trace_mark(trace, idx, 1);   // before any write is visible
        for (int i = lane; i < k; i += 32) {
            int jj = col[b + i];
            float xx = val ? val[b + i] : 1.0f;
            __stcg(w + jj, __fsub_rn(__ldcg(w + jj), __fmul_rn(c, xx)));
        }
    }
    __syncwarp();
}

// ---------------------------------------------------------------- level-synchronous engine
// Persistent cooperative kernel: level l's examples are spread over all
// warps, a grid barrier closes the level (the read barrier of the next BSP
// step and the write barrier of this one, Algorithm 2a per level).
template <int R>
__global__ __launch_bounds__(THREADS) void k_sgd_levels(int32_t n_rows, const int64_t *__restrict__ row_ptr,
                                                        const int32_t *__restrict__ col, const float *__restrict__ val,
                                                        const float *__restrict__ y, const int32_t *__restrict__ order,
                                                        const int64_t *__restrict__ level_ptr, const LevelCtl *ctl,
                                                        float *w, int loss, float eta, int epochs, GridBarrier *bar,
                                                        int *status, uint64_t timeout, uint64_t *trace)
{
    if (read_status(status)) return;
    const int L = ctl->n_levels;
    const int gw = (int)(((int64_t)blockIdx.x * blockDim.x + threadIdx.x) >> 5);
    const int nw = (int)(((int64_t)gridDim.x * blockDim.x) >> 5);
    for (int ep = 0; ep < epochs; ++ep)
        for (int l = 0; l < L; ++l) {
            const int64_t b = level_ptr[l], e = level_ptr[l + 1];
            for (int64_t i = b + gw; i < e; i += nw) {
                const int t = order[i];
                if (t < 0 || t >= n_rows) {      // cannot happen with a consistent schedule
                    set_status(status, PDB_EFAULT);
                    continue;
                }
                sgd_example<R>(t, row_ptr, col, val, y, w, loss, eta, trace, (int64_t)ep * n_rows + t);
            }
            if (!grid_sync(bar, status, timeout)) return;
        }
}

// ---------------------------------------------------------------- ready-counter dataflow engine
// The read protocol of Section 5 per feature.  Feature j's record holds its
// weight and its iteration number (version) in one aligned 64-bit word:
// rec[j] = bits(w_j) | version_j << 32.  The occurrence of j with rank r
// (its gate) may read w_j once version_j == r -- one relaxed 64-bit load
// both checks the version and returns the weight written with it (Read
// Constraint: the previous writer is done) -- and publishes the new weight
// together with version r + 1 in one 64-bit store (Write Constraint: its own
// read, the only read of that version, came first).  Both halves travel in
// one single-copy-atomic access, so no fence is needed.
// All epochs run in one launch, pipelined: rank r of epoch e waits for version
// e * n_rows + r (a rank is below n_rows), and the last occurrence of j in an
// epoch (GATE_LAST) publishes (e + 1) * n_rows, so the next epoch's first
// occurrence of j starts as soon as that write lands -- not at a kernel
// boundary (exact by Theorem 2: per feature the order is still the data order,
// epoch after epoch).  Versions count modulo 2^32: two that are equal lie
// 2^31 examples or more apart, far more than are ever in flight.
// Examples are taken in data order (epoch-major) from a ticket counter,
// `chunk` consecutive ones at a time and run in order by the warp that took
// them, so the oldest unfinished example never waits on a younger one and
// the kernel cannot deadlock whatever the number of resident warps.
__device__ __forceinline__ unsigned long long ld_rec(const unsigned long long *p)
{
    unsigned long long v;
    asm volatile("ld.relaxed.gpu.global.b64 %0, [%1];" : "=l"(v) : "l"(p) : "memory");
    return v;
}
__device__ __forceinline__ void st_rec(unsigned long long *p, float w, unsigned version)
{
    unsigned long long v = (unsigned long long)__float_as_uint(w) | ((unsigned long long)version << 32);
    asm volatile("st.relaxed.gpu.global.b64 [%0], %1;" ::"l"(p), "l"(v) : "memory");
}

// Gathers w for the lane's elements (bit r of `pending`: the lane has element r),
// waiting until each record carries the wanted version; called by the whole
// warp.  False when the wait gave up (timeout or a failure elsewhere recorded in
// status).  The loop is the warp's, not each lane's: lanes that left it one by
// one would stay apart, and every shuffle after it would first have to bring
// them together again (~280 cycles each, measured).
template <int R>
__device__ __forceinline__ bool gather_ready(const unsigned long long *rec, const int *j, const unsigned *want,
                                             unsigned pending, float *wv, int *status, uint64_t timeout)
{
    uint64_t t0 = 0;
    for (unsigned spins = 0;; ++spins) {
#pragma unroll
        for (int r = 0; r < R; ++r) {
            unsigned long long v = 0;
            if (pending & (1u << r)) v = ld_rec(rec + j[r]);
            const bool hit = (pending & (1u << r)) && (unsigned)(v >> 32) == want[r];
            wv[r] = hit ? __uint_as_float((unsigned)v) : wv[r];
            pending &= hit ? ~(1u << r) : ~0u;
        }
        if (!__any_sync(FULL, pending)) return true;
        if ((spins & 31u) == 31u) {
            const uint64_t now = globaltimer();
            if (spins == 31u) t0 = now;
            bool stop = read_status(status) != 0;
            if (!stop && now - t0 > timeout) {
                set_status(status, PDB_ETIMEOUT);
                stop = true;
            }
            if (__any_sync(FULL, stop)) return false;
        }
    }
}

// An example of more ids than a warp's registers hold: wait and gather L elements per
// lane at a time, then a second pass (this example owns its features until it
// writes them, so re-reading the records returns the same weights).  Two epochs with
// one element per lane at a time, each waited for by the whole warp, and with eight:
// 3000 rows of 500 uniform ids over 60000 features 87.7 and 47.9 ms, 5000 of 1000 over
// 20M 32.8 and 20.0, 1551 of 293 zipf-like ids over 969 features 23.5 and 20.5.
template <int L>
__device__ __forceinline__ bool long_example(int64_t b, int k, float yt, unsigned base, unsigned next_base,
                                        const int32_t *__restrict__ col, const float *__restrict__ val,
                                        const uint32_t *__restrict__ gate, unsigned long long *rec, int loss, float eta,
                                        int *status, uint64_t timeout, uint64_t *trace, int64_t idx)
{
    const int lane = threadIdx.x & 31;
    float acc = 0.0f;
    for (int i0 = 0; i0 < k; i0 += 32 * L) {
        int j[L];
        float x[L], wv[L];
        unsigned want[L], have = 0;
#pragma unroll
        for (int r = 0; r < L; ++r) {
            const int i = i0 + r * 32 + lane;
            have |= i < k ? 1u << r : 0u;
            j[r] = i < k ? col[b + i] : 0;
            x[r] = i < k ? (val ? val[b + i] : 1.0f) : 0.0f;
            want[r] = base + (i < k ? gate[b + i] & GATE_RANK : 0u);
            wv[r] = 0.0f;
        }
        if (!gather_ready<L>(rec, j, want, have, wv, status, timeout)) return false;
#pragma unroll
        for (int r = 0; r < L; ++r)
            if (have >> r & 1u) acc = __fmaf_rn(wv[r], x[r], acc);
    }
    trace_mark(trace, idx, 0);
    const float m = warp_combine_latency(acc);
    const float c = dev_step(loss, m, yt, eta);
    trace_mark(trace, idx, 1);   // before any write is visible
    for (int i = lane; i < k; i += 32) {
        const int jj = col[b + i];
        const float xx = val ? val[b + i] : 1.0f;
        const uint32_t g = gate[b + i];
        const float wo = __uint_as_float((unsigned)ld_rec(rec + jj));
        st_rec(rec + jj, __fsub_rn(wo, __fmul_rn(c, xx)), (g & GATE_LAST) ? next_base : base + (g & GATE_RANK) + 1u);
    }
    return true;
}

// The widest kernel's, apart from its code: inlined there it slows the shorter rows
// (20000 rows of 256 ids over 20M features 0.45 -> 0.55 ms).  The narrower kernels
// meet no such row (they are chosen by the longest one).
__device__ __noinline__ bool long_example_apart(int64_t b, int k, float yt, unsigned base, unsigned next_base,
                                                const int32_t *__restrict__ col, const float *__restrict__ val,
                                                const uint32_t *__restrict__ gate, unsigned long long *rec, int loss,
                                                float eta, int *status, uint64_t timeout, uint64_t *trace, int64_t idx)
{
    return long_example<8>(b, k, yt, base, next_base, col, val, gate, rec, loss, eta, status, timeout, trace, idx);
}

// one example under the ready protocol; false when a wait gave up
template <int R>
__device__ __forceinline__ bool ready_example(int t, unsigned base, unsigned next_base,
                                              const int64_t *__restrict__ row_ptr,
                                              const int32_t *__restrict__ col, const float *__restrict__ val,
                                              const float *__restrict__ y, const uint32_t *__restrict__ gate,
                                              unsigned long long *rec, int loss, float eta, int *status,
                                              uint64_t timeout, uint64_t *trace, int64_t idx)
{
    const int lane = threadIdx.x & 31;
    const int64_t b = row_ptr[t];
    const int k = (int)(row_ptr[t + 1] - b);
    const float yt = y[t];
    if (k <= 32 * R) {
        int j[R];
        float x[R], wv[R];
        unsigned want[R], next[R], have = 0;
#pragma unroll
        for (int r = 0; r < R; ++r) {
            int i = r * 32 + lane;
            have |= i < k ? 1u << r : 0u;
            j[r] = i < k ? col[b + i] : 0;
            x[r] = i < k ? (val ? val[b + i] : 1.0f) : 0.0f;
            uint32_t g = i < k ? gate[b + i] : 0u;
            want[r] = base + (g & GATE_RANK);
            next[r] = (g & GATE_LAST) ? next_base : want[r] + 1u;
            wv[r] = 0.0f;
        }
        if (!gather_ready<R>(rec, j, want, have, wv, status, timeout)) return false;
        trace_mark(trace, idx, 0);
        float acc = 0.0f;
#pragma unroll
        for (int r = 0; r < R; ++r)
            if (r * 32 + lane < k) acc = __fmaf_rn(wv[r], x[r], acc);
        const float m = warp_combine_latency(acc);
        const float c = dev_step(loss, m, yt, eta);
        trace_mark(trace, idx, 1);   // before any write is visible
#pragma unroll
        for (int r = 0; r < R; ++r)
            if (r * 32 + lane < k) st_rec(rec + j[r], __fsub_rn(wv[r], __fmul_rn(c, x[r])), next[r]);
        return true;
    }
    if constexpr (R < 8)
        return long_example<1>(b, k, yt, base, next_base, col, val, gate, rec, loss, eta, status, timeout, trace, idx);
    else
        return long_example_apart(b, k, yt, base, next_base, col, val, gate, rec, loss, eta, status, timeout, trace, idx);
}

template <int R>
__global__ __launch_bounds__(THREADS) void k_sgd_ready(int32_t n_rows, const int64_t *__restrict__ row_ptr,
                                                       const int32_t *__restrict__ col, const float *__restrict__ val,
                                                       const float *__restrict__ y, const uint32_t *__restrict__ gate,
                                                       unsigned long long *rec, int loss, float eta, int epochs,
                                                       unsigned long long *ticket, int chunk, int *status,
                                                       uint64_t timeout, uint64_t *trace)
{
    if (read_status(status)) return;
    const int lane = threadIdx.x & 31;
    const int64_t total = (int64_t)epochs * n_rows;     // examples of all epochs, epoch-major
    for (;;) {
        unsigned long long tk = 0;
        if (lane == 0) tk = atomicAdd(ticket, (unsigned long long)chunk);
        tk = __shfl_sync(FULL, tk, 0);
        if (tk >= (unsigned long long)total) return;
        const int64_t t1 = min64(total, (int64_t)tk + chunk);
        for (int64_t tg = (int64_t)tk; tg < t1; ++tg) {
            const int64_t e = tg / n_rows;
            const unsigned base = (unsigned)e * (unsigned)n_rows;
            if (!ready_example<R>((int)(tg - e * n_rows), base, base + (unsigned)n_rows, row_ptr, col, val, y, gate, rec,
                                  loss, eta, status, timeout, trace, tg))
                return;
        }
    }
}

// rec[j] = (w_j, version 0 of the first epoch) before the first epoch; w_j
// back after the last
__global__ void k_pack(const float *__restrict__ w, int64_t n, unsigned long long *__restrict__ rec, const int *status)
{
    if (read_status(status)) return;
    for (int64_t i = (int64_t)blockIdx.x * blockDim.x + threadIdx.x; i < n; i += (int64_t)gridDim.x * blockDim.x)
        rec[i] = (unsigned long long)__float_as_uint(w[i]);
}

__global__ void k_unpack(const unsigned long long *__restrict__ rec, int64_t n, float *__restrict__ w,
                         const int *status)
{
    if (read_status(status)) return;
    for (int64_t i = (int64_t)blockIdx.x * blockDim.x + threadIdx.x; i < n; i += (int64_t)gridDim.x * blockDim.x)
        w[i] = __uint_as_float((unsigned)rec[i]);
}

// ---------------------------------------------------------------- BSP
// Per batch two launches: k_bsp_coef (the reads) and k_bsp_apply (the writes).
// A batch's launches follow each other with programmatic dependence: a kernel
// starts while the one before it drains, reads what no batch writes (row
// bounds, ids, values, rows of pairs), and waits here before it reads what the
// one before wrote.  Without that launch attribute both are no-ops.
__device__ __forceinline__ void launch_next() { asm volatile("griddepcontrol.launch_dependents;" ::: "memory"); }
__device__ __forceinline__ void wait_previous() { asm volatile("griddepcontrol.wait;" ::: "memory"); }

// loads that stay where they are written: the compiler may move a load of
// read-only data down to its use, behind the work that should hide it
__device__ __forceinline__ int32_t ld_here(const int32_t *p)
{
    int32_t v;
    asm volatile("ld.global.s32 %0, [%1];" : "=r"(v) : "l"(p) : "memory");
    return v;
}
__device__ __forceinline__ float ld_here(const float *p)
{
    float v;
    asm volatile("ld.global.cg.f32 %0, [%1];" : "=f"(v) : "l"(p) : "memory");
    return v;
}

// margin of example t at the current w (all lanes return the same value); rows
// longer than 32 ids load BSP_M elements per lane at a time, the next ones' ids
// and values while these ones' weights are on their way
constexpr int BSP_M = 8;
__device__ __forceinline__ float margin(int t, const int64_t *__restrict__ row_ptr, const int32_t *__restrict__ col,
                                        const float *__restrict__ val, const float *w)
{
    const int lane = threadIdx.x & 31;
    const int64_t b = row_ptr[t];
    const int k = (int)(row_ptr[t + 1] - b);
    float acc = 0.0f;
    if (k <= 32) {
        int j0 = 0;
        float x0 = 1.0f;
        if (lane < k) {
            j0 = ld_here(col + b + lane);
            if (val) x0 = ld_here(val + b + lane);
        }
        wait_previous();
        if (lane < k) acc = __fmaf_rn(__ldcg(w + j0), x0, acc);
        return warp_combine(acc);
    }
    int j[BSP_M];
    float x[BSP_M], wv[BSP_M], xc[BSP_M];
    auto load = [&](int base) {
#pragma unroll
        for (int u = 0; u < BSP_M; ++u) {
            const int i = min(base + 32 * u + lane, k - 1);      // past the end: the last element, not added
            j[u] = ld_here(col + b + i);
            x[u] = val ? ld_here(val + b + i) : 1.0f;
        }
    };
    load(0);
    wait_previous();
    for (int base = 0; base < k; base += 32 * BSP_M) {
#pragma unroll
        for (int u = 0; u < BSP_M; ++u) {
            wv[u] = __ldcg(w + j[u]);
            xc[u] = x[u];
        }
        if (base + 32 * BSP_M < k) load(base + 32 * BSP_M);
#pragma unroll
        for (int u = 0; u < BSP_M; ++u)
            if (base + 32 * u + lane < k) acc = __fmaf_rn(wv[u], xc[u], acc);
    }
    return warp_combine(acc);
}

// The write half of a batch works on its pairs [s0, s1), sorted by (feature,
// example): feature j's terms c_i * x_ij form one run, added in ascending
// example order from +0; then w_j = w_j - sum.  The batch's rows start at r0
// and coef holds their coefficients.  Positions are below 2^31; unsigned, so
// that looking some turns ahead does not overflow.
struct BspPairs {
    uint32_t s1;            // the batch's end
    int32_t r0, rows;
    const int32_t *__restrict__ col, *__restrict__ row;
    const float *__restrict__ val;
    const float *coef;
};

// the coefficient of a pair's example (`bad` set for a row outside the batch:
// cannot happen with a consistent batch sort)
__device__ __forceinline__ float bsp_coef_of(const BspPairs &P, int32_t row, bool &bad)
{
    const int32_t i = row - P.r0;
    const bool in = i >= 0 && i < P.rows;
    bad |= !in;
    return ld_here(P.coef + (in ? i : 0));
}
// the same when `on`, else 0 without an access
__device__ __forceinline__ float bsp_coef_if(const BspPairs &P, int32_t row, bool on, bool &bad)
{
    const int32_t i = row - P.r0;
    const bool in = i >= 0 && i < P.rows;
    bad |= on && !in;
    float v;
    asm volatile("{\n\t.reg .pred p;\n\tsetp.ne.s32 p, %2, 0;\n\tmov.f32 %0, 0f00000000;\n\t@p ld.global.cg.f32 %0, [%1];\n\t}"
                 : "=f"(v)
                 : "l"(P.coef + (in ? i : 0)), "r"((int)on)
                 : "memory");
    return v;
}

// A run longer than BSP_LONG terms is summed by a block: warp 0 adds, the
// others make the products.
constexpr int BSP_LONG = 16;
constexpr int BSP_THREADS = 128;
constexpr int BSP_BLOCKS = 8;                       // per SM
constexpr int BSP_U = 8;                            // terms per producing thread and stage
constexpr int BSP_STAGE = (BSP_THREADS - 32) * BSP_U;
constexpr int BSP_ADDS = 192;                       // terms the adding warp takes between two loop branches

// The sum of the `len` terms from pair q on, by the whole block; the result is
// warp 0's.  The sum is a chain of dependent additions (4 cycles each), so one
// warp does nothing else: it adds a stage of products from shared memory, 16
// bytes per load, every lane the same, while the other warps form the next
// stage's (rows loaded one stage earlier still).  A stage's terms past the
// run's end are -0, which changes no sum.
__device__ __forceinline__ float block_run_sum(const BspPairs &P, uint32_t q, uint32_t len, float (*buf)[BSP_STAGE],
                                               bool &bad)
{
    const int t = (int)threadIdx.x - 32;            // producer, < 0: the adding warp
    const uint32_t end = q + len, stages = (len + BSP_STAGE - 1) / BSP_STAGE;
    int32_t row[BSP_U];
    auto rows_of = [&](uint32_t k) {
#pragma unroll
        for (int u = 0; u < BSP_U; ++u)
            row[u] = ld_here(P.row + min(q + k * BSP_STAGE + u * (BSP_THREADS - 32) + t, end - 1));
    };
    auto produce = [&](uint32_t k) {                // stage k, its rows in row[]
        float v[BSP_U], c[BSP_U];
#pragma unroll
        for (int u = 0; u < BSP_U; ++u)
            v[u] = ld_here(P.val + min(q + k * BSP_STAGE + u * (BSP_THREADS - 32) + t, end - 1));
        if (k == 0) wait_previous();                // the coefficients are the kernel before's
#pragma unroll
        for (int u = 0; u < BSP_U; ++u) c[u] = bsp_coef_of(P, row[u], bad);
        if (k + 1 < stages) rows_of(k + 1);
#pragma unroll
        for (int u = 0; u < BSP_U; ++u) {
            const int i = u * (BSP_THREADS - 32) + t;
            buf[k & 1][i] = k * BSP_STAGE + i < len ? __fmul_rn(c[u], v[u]) : -0.0f;
        }
    };
    float delta = 0.0f;
    if (t >= 0) {
        rows_of(0);
        produce(0);
    } else {
        wait_previous();
    }
    __syncthreads();
    for (uint32_t k = 0; k < stages; ++k) {
        if (t >= 0) {
            if (k + 1 < stages) produce(k + 1);
        } else {
            const float4 *b4 = reinterpret_cast<const float4 *>(buf[k & 1]);
            const int n = (int)min(len - k * BSP_STAGE, (uint32_t)BSP_STAGE);
#pragma unroll 1
            for (int i = 0; i < n; i += BSP_ADDS, b4 += BSP_ADDS / 4)
#pragma unroll
                for (int e = 0; e < BSP_ADDS / 4; ++e) {
                    const float4 f = b4[e];
                    delta = __fadd_rn(__fadd_rn(__fadd_rn(__fadd_rn(delta, f.x), f.y), f.z), f.w);
                }
        }
        __syncthreads();
    }
    return delta;
}
static_assert(BSP_STAGE % BSP_ADDS == 0, "the adding warp reads whole groups");

// The next CH terms of feature j's run from q, added to delta (loads first,
// then the dependent adds).  Returns whether the run may continue past them.
template <int CH>
__device__ __forceinline__ bool thread_run_chunk(const BspPairs &P, int32_t j, uint32_t &q, float &delta, bool &bad)
{
    int32_t jj[CH], rr[CH];
    float xx[CH], cc[CH];
#pragma unroll
    for (int u = 0; u < CH; ++u) {
        const bool in = q + u < P.s1;
        jj[u] = in ? P.col[q + u] : -1;
        rr[u] = in ? P.row[q + u] : P.r0;
        xx[u] = in ? P.val[q + u] : 0.0f;
    }
    bool more = true;
    int n = 0;
#pragma unroll
    for (int u = 0; u < CH; ++u) {
        more = more && jj[u] == j;
        n += more;
        cc[u] = bsp_coef_if(P, rr[u], more, bad);
    }
#pragma unroll
    for (int u = 0; u < CH; ++u)
        if (u < n) delta = __fadd_rn(delta, __fmul_rn(cc[u], xx[u]));
    q += CH;
    return more;
}

// BSP_R of the short runs (at most BSP_LONG terms): i and i + step of the n of a
// batch.  The first two terms of each (most runs hold one or two) and its weight
// are loaded together, the rest term by term.  A coefficient is a random access
// like the weight, so it is loaded for the run's own terms only: loading the
// second one always cost half of the time of a batch of single terms.  Measured,
// ms per epoch, with that load / without it and 1, 2, 4 runs at once: 10000 rows of
// 1000 uniform ids over 50M features, batches of 4096: 0.632 / 0.432, 0.427, 0.412;
// 400k rows of 50 over 10M, batches of 65536: 0.472 / 0.425, 0.393, 0.377; 200k rows
// of 20 zipf(1.0)-like ids, batches of 256: - / 4.71, 4.71, 5.26.
constexpr int BSP_R = 2;
__device__ __forceinline__ void short_runs(const BspPairs &P, const int32_t *__restrict__ runs, uint32_t i, uint32_t step,
                                           uint32_t n, float *w, bool &bad)
{
    uint32_t q[BSP_R];
    int32_t j[BSP_R], row[BSP_R], row2[BSP_R];
    float x[BSP_R], x2[BSP_R], wj[BSP_R], delta[BSP_R];
    bool second[BSP_R];
#pragma unroll
    for (int u = 0; u < BSP_R; ++u) q[u] = i + u * step < n ? (uint32_t)runs[i + u * step] : P.s1;
#pragma unroll
    for (int u = 0; u < BSP_R; ++u) {
        const bool in = q[u] < P.s1, in2 = q[u] + 1 < P.s1;
        j[u] = in ? P.col[q[u]] : -1;
        second[u] = in2 && P.col[q[u] + 1] == j[u];
        row[u] = in ? P.row[q[u]] : P.r0;
        row2[u] = in2 ? P.row[q[u] + 1] : P.r0;
        x[u] = in ? P.val[q[u]] : 0.0f;
        x2[u] = in2 ? P.val[q[u] + 1] : 0.0f;
    }
#pragma unroll
    for (int u = 0; u < BSP_R; ++u) {
        wj[u] = j[u] >= 0 ? __ldcg(w + j[u]) : 0.0f;
        const float c = bsp_coef_if(P, row[u], j[u] >= 0, bad), c2 = bsp_coef_if(P, row2[u], second[u], bad);
        delta[u] = __fadd_rn(0.0f, __fmul_rn(c, x[u]));
        if (second[u]) delta[u] = __fadd_rn(delta[u], __fmul_rn(c2, x2[u]));
    }
#pragma unroll
    for (int u = 0; u < BSP_R; ++u) {
        if (second[u]) {
            q[u] += 2;
            while (thread_run_chunk<4>(P, j[u], q[u], delta[u], bad)) {}
        }
        if (j[u] >= 0) __stcg(w + j[u], __fsub_rn(wj[u], delta[u]));
    }
}

// The runs of every batch, in no particular order: their first pairs at
// runs[bptr[b] ..] (at most BSP_LONG terms) and, for longer ones, the first pair
// and the length, two words each, backwards from runs[bptr[b + 1] - 1] (a long
// run has more than two pairs, so the two lists never meet); counts in n_runs[b]
// (short, long; zeroed before).  skey: the batch of each pair (null: one batch).
// A block's turn is a chain of waits (pairs, bounds, places), so what bounds this is
// how much one warp has in flight and how little it loads: each pair's feature once,
// its neighbours' by shuffles.  20M pairs in one batch / in seven: 97 / 109 us with
// six loads per pair and a reservation per warp, 48 / 52 so (four blocks per SM; five
// or more spill).
static_assert(BSP_LONG == 16, "the pair a long run's length ahead is in the other half of the warp");
__global__ __launch_bounds__(256, 4) void k_bsp_runs(const uint32_t *__restrict__ skey, const int32_t *__restrict__ bcol,
                           const int64_t *__restrict__ bptr, int64_t nnz, int32_t *__restrict__ runs, uint2 *n_runs,
                           const int *status)
{
    if (read_status(status)) return;
    constexpr int E = 8;                // 256 pairs per warp and turn
    __shared__ unsigned s_n[2][8];      // short and long runs of the block's warps, then where each puts its own
    const int lane = threadIdx.x & 31, warp = threadIdx.x >> 5;
    const uint32_t n = (uint32_t)nnz, stride = gridDim.x * 256u * E;       // (no overflow: n < 2^31, stride < 2^24)
    for (uint32_t base0 = blockIdx.x * 256u * E; base0 < n; base0 += stride) {
        const uint32_t base = base0 + (uint32_t)warp * 32u * E;
        // the features of the warp's pairs, of the one before them and of the 16 after
        int32_t j[E + 1], prev = base > 0 && base <= n ? bcol[base - 1] : -1;
#pragma unroll
        for (int e = 0; e <= E; ++e) {
            const uint32_t s = base + 32u * e + lane;
            j[e] = s < n && (e < E || lane < BSP_LONG) ? bcol[s] : -1;
        }
        // the batches of the warp's pairs, one after the other.  A block whose pairs are
        // all of one batch (nearly always) reserves its places in the lists at once, since
        // a batch's counter is one address.
        const bool one_batch = !skey || skey[base0] == skey[min(n, base0 + 256u * E) - 1];
        const uint32_t b_first = skey ? skey[one_batch ? base0 : min(base, n - 1)] : 0u;
        const uint32_t b_last = one_batch ? b_first : skey[min(n, base + 32u * E) - 1];
        for (uint32_t bb = b_first; bb <= b_last; ++bb) {
            const uint32_t b0 = (uint32_t)bptr[bb], b1 = (uint32_t)bptr[bb + 1];
            unsigned sm[E], lm[E], n_s = 0, n_l = 0;
            int32_t last = prev, half = __shfl_xor_sync(FULL, j[0], BSP_LONG);
#pragma unroll
            for (int e = 0; e < E; ++e) {
                const uint32_t s = base + 32u * e + lane;
                const int32_t turn = __shfl_sync(FULL, j[e], (lane + 31) & 31), next = __shfl_xor_sync(FULL, j[e + 1], BSP_LONG);
                const int32_t before = lane ? turn : last, far = lane < BSP_LONG ? half : next;
                last = turn;                   // lane 0: the last of these 32
                half = next;
                const bool start = s >= b0 && s < b1 && (s == b0 || before != j[e]);
                const bool is_long = start && s + BSP_LONG < b1 && far == j[e];
                sm[e] = __ballot_sync(FULL, start && !is_long);
                lm[e] = __ballot_sync(FULL, is_long);
            }
#pragma unroll
            for (int e = 0; e < E; ++e) {
                n_s += __popc(sm[e]);
                n_l += __popc(lm[e]);
            }
            unsigned at_s = 0, at_l = 0;
            if (one_batch) {
                __syncthreads();               // the turn before has read its places
                if (lane == 0) {
                    s_n[0][warp] = n_s;
                    s_n[1][warp] = n_l;
                }
                __syncthreads();
                if (threadIdx.x < 2) {         // one thread per counter
                    unsigned all = 0, at[8];
#pragma unroll
                    for (int i = 0; i < 8; ++i) {
                        at[i] = all;
                        all += s_n[threadIdx.x][i];
                    }
                    const unsigned place = all ? atomicAdd(threadIdx.x ? &n_runs[bb].y : &n_runs[bb].x, all) : 0u;
#pragma unroll
                    for (int i = 0; i < 8; ++i) s_n[threadIdx.x][i] = place + at[i];
                }
                __syncthreads();
                at_s = s_n[0][warp];
                at_l = s_n[1][warp];
            } else {
                if (lane == 0 && n_s) at_s = atomicAdd(&n_runs[bb].x, n_s);
                if (lane == 0 && n_l) at_l = atomicAdd(&n_runs[bb].y, n_l);
                at_s = __shfl_sync(FULL, at_s, 0);
                at_l = __shfl_sync(FULL, at_l, 0);
            }
#pragma unroll
            for (int e = 0; e < E; ++e) {
                const uint32_t s = base + 32u * e + lane;
                if (sm[e] >> lane & 1u) runs[b0 + at_s + __popc(sm[e] & lanemask_lt())] = (int32_t)s;
                at_s += __popc(sm[e]);
            }
            if (n_l == 0) continue;
#pragma unroll
            for (int e = 0; e < E; ++e) {
                const uint32_t s = base + 32u * e + lane;
                if (lm[e] >> lane & 1u) {
                    // the run's length: doubling steps, then a binary search (the batch's
                    // pairs are sorted by feature)
                    uint32_t lo = s + BSP_LONG, step = BSP_LONG, hi = lo + step;     // bcol[lo] == j
                    while (hi < b1 && bcol[hi] == j[e]) {
                        lo = hi;
                        step *= 2;
                        hi = lo + step;
                    }
                    hi = min(hi, b1);
                    while (hi - lo > 1) {
                        const uint32_t mid = lo + ((hi - lo) >> 1);
                        if (bcol[mid] == j[e])
                            lo = mid;
                        else
                            hi = mid;
                    }
                    const uint32_t at = b1 - 2 * (at_l + __popc(lm[e] & lanemask_lt()) + 1);
                    runs[at] = (int32_t)s;
                    runs[at + 1] = (int32_t)(lo + 1 - s);
                }
                at_l += __popc(lm[e]);
            }
        }
    }
}

__global__ void k_bsp_keys(const int32_t *__restrict__ csc_pos, const int32_t *__restrict__ row_of, int64_t nnz,
                           uint32_t batch, uint32_t *__restrict__ key, const int *status)
{
    if (read_status(status)) return;
    for (int64_t s = (int64_t)blockIdx.x * blockDim.x + threadIdx.x; s < nnz; s += (int64_t)gridDim.x * blockDim.x)
        key[s] = (uint32_t)row_of[csc_pos[s]] / batch;
}

__global__ void k_bsp_gather(const int32_t *__restrict__ bpos, const int32_t *__restrict__ col,
                             const float *__restrict__ val, const int32_t *__restrict__ row_of, int64_t nnz,
                             int32_t *__restrict__ bcol, int32_t *__restrict__ brow, float *__restrict__ bval,
                             const int *status)
{
    if (read_status(status)) return;
    for (int64_t s = (int64_t)blockIdx.x * blockDim.x + threadIdx.x; s < nnz; s += (int64_t)gridDim.x * blockDim.x) {
        int32_t p = bpos[s];
        bcol[s] = col[p];
        brow[s] = row_of[p];
        bval[s] = val ? val[p] : 1.0f;
    }
}

__global__ void k_bsp_one_batch(int64_t *__restrict__ bptr, int64_t nnz)
{
    bptr[0] = 0;
    bptr[1] = nnz;
}

// ---- Algorithm 2a split over data-parallel ranks (pdb_bsp_plan / coef / apply)
// c_i = eta * dloss/dm(m_i(w), y_i) for the rows [r0, r1), one warp per example,
// w the weights of the batch start (the read half of the step)
__global__ __launch_bounds__(256, 5) void k_bsp_coef(int64_t r0, int64_t r1, const int64_t *__restrict__ row_ptr,
                           const int32_t *__restrict__ col, const float *__restrict__ val,
                           const float *__restrict__ y, const float *w, int loss, float eta, float *__restrict__ coef,
                           const int *status)
{
    launch_next();
    if (read_status(status)) {
        wait_previous();        // a kernel that is done leaves nothing before it running
        return;
    }
    const int lane = threadIdx.x & 31;
    const int64_t gw = ((int64_t)blockIdx.x * blockDim.x + threadIdx.x) >> 5;
    const int64_t nw = ((int64_t)gridDim.x * blockDim.x) >> 5;
    for (int64_t t = r0 + gw; t < r1; t += nw) {
        const float yt = y[t];
        const float m = margin((int)t, row_ptr, col, val, w);       // waits for the batch before
        if (lane == 0) coef[t - r0] = __fmul_rn(eta, dev_grad(loss, m, yt));
    }
}

// The write half of batch bi: coef holds the whole batch's coefficients (rows
// r0.. in order).  Long runs one per block; short ones BSP_R per thread, on the
// blocks without a long one when those are most.
//
// What bounds it: the longest run's additions (3000 terms of the hottest
// feature in a batch of 4096 zipf(1.0) examples: ~6 us).  Measured, both
// launches of such a batch: 12 us, against 41 in one cooperative kernel whose
// warps loaded 32 terms, shuffled them out and added them before the next 32
// arrived (27 cycles per term), with two grid barriers of ~3 us each; on 5000
// dense examples of 960 features 37 us per batch against 113.  One warp doing
// both loads and additions took 6 cycles per term alone and 13 with every SM
// doing so.
//
// The weights are read and written through L2 only, never a line kept in L1:
// this block may already sit on an SM while blocks of the batch before there
// still read and write other weights of the same lines.
__global__ __launch_bounds__(BSP_THREADS, BSP_BLOCKS) void k_bsp_apply(
    int64_t bi, const int64_t *__restrict__ bptr, int32_t r0, int32_t rows, const int32_t *__restrict__ bcol,
    const int32_t *__restrict__ brow, const float *__restrict__ bval, const int32_t *__restrict__ runs,
    const uint2 *__restrict__ n_runs, const float *coef, float *w, int *status)
{
    __shared__ __align__(16) float s_buf[2][BSP_STAGE];
    launch_next();
    if (read_status(status)) {
        wait_previous();        // as in k_bsp_coef
        return;
    }
    const int64_t s0 = bptr[bi], s1 = bptr[bi + 1];
    const uint2 n = n_runs[bi];
    const BspPairs P = {(uint32_t)s1, r0, rows, bcol, brow, bval, coef};
    bool bad = false;
    for (uint32_t i = blockIdx.x; i < n.y; i += gridDim.x) {
        const int64_t at = s1 - 2 * ((int64_t)i + 1);
        const uint32_t q = (uint32_t)runs[at], len = (uint32_t)runs[at + 1];
        const float delta = block_run_sum(P, q, len, s_buf, bad);
        if (threadIdx.x == 0) {
            const int32_t j = bcol[q];
            __stcg(w + j, __fsub_rn(__ldcg(w + j), delta));
        }
    }
    wait_previous();
    const uint32_t b0 = n.y < gridDim.x / 2 ? n.y : 0;
    if (blockIdx.x >= b0) {
        const uint32_t step = (gridDim.x - b0) * BSP_THREADS;
        for (uint32_t i = (blockIdx.x - b0) * BSP_THREADS + threadIdx.x; i < n.x; i += BSP_R * step)
            short_runs(P, runs + s0, i, step, n.x, w, bad);
    }
    if (bad) set_status(status, PDB_EFAULT);   // cannot happen with a consistent batch order
}

__global__ void k_eval_grad(const float *__restrict__ m, const float *__restrict__ y, float *__restrict__ out,
                            int64_t n, int loss)
{
    for (int64_t i = (int64_t)blockIdx.x * blockDim.x + threadIdx.x; i < n; i += (int64_t)gridDim.x * blockDim.x)
        out[i] = dev_grad(loss, m[i], y[i]);
}

__global__ void k_eval_expf(const float *__restrict__ x, float *__restrict__ out, int64_t n)
{
    for (int64_t i = (int64_t)blockIdx.x * blockDim.x + threadIdx.x; i < n; i += (int64_t)gridDim.x * blockDim.x)
        out[i] = dev_expf(x[i]);
}

// Registers per lane for the example's elements: the smallest of 2, 4, 8
// that holds the longest row in registers (longer rows take the two-pass
// path).  The longest row is recorded by the conflict build; this waits for
// that build to finish if it has not.
int register_width(const pdb_conflicts *c)
{
    if (cudaEventSynchronize(c->ev1) != cudaSuccess) {
        cudaGetLastError();
        return 8;
    }
    const int longest = c->h_info[2];
    return longest <= 64 ? 2 : longest <= 128 ? 4 : 8;
}

// The pairs of c in (batch, feature, example) order: feature, example and value
// of each, where each batch's pairs start, and each batch's runs (enqueued on
// s).  The CSC order is already (feature, example), so a single batch needs no
// sort.
int bsp_sort(pdb_conflicts *c, const float *val, int64_t batch, int64_t n_batches, int32_t *bcol, int32_t *brow,
             float *bval, int64_t *bptr, int32_t *runs, uint2 *n_runs, cudaStream_t s)
{
    const int64_t nnz = c->nnz;
    const int rf = fill_words(n_runs, 0u, sizeof(uint2) * std::max<int64_t>(n_batches, 1), s);
    if (rf != PDB_OK) return rf;
    if (nnz == 0) return fill_words(bptr, 0u, sizeof(int64_t) * (n_batches + 1), s);
    uint32_t *key = nullptr, *skey = nullptr, *tkey = nullptr;
    int32_t *bpos = nullptr, *tval = nullptr;
    Block scratch;
    int rc = ensure_row_of(c, s);
    if (n_batches > 1) {
        rc = rc ? rc : alloc_block(scratch, {{(void **)&key, sizeof(uint32_t) * nnz},
                                              {(void **)&skey, sizeof(uint32_t) * nnz},
                                              {(void **)&tkey, sizeof(uint32_t) * nnz},
                                              {(void **)&bpos, sizeof(int32_t) * nnz},
                                              {(void **)&tval, sizeof(int32_t) * nnz}}, s);
        if (rc == PDB_OK) {
            k_bsp_keys<<<grid_1d(nnz), 256, 0, s>>>(c->csc_pos, c->row_of, nnz, (uint32_t)batch, key, c->status);
            note_launch();
            // stable by batch: inside a batch the feature-major CSC order survives
            rc = radix_sort(key, c->csc_pos, skey, bpos, tkey, tval, nnz, bits_for(n_batches - 1), c->status, s);
            rc = rc ? rc : segment_bounds(skey, nnz, n_batches, nullptr, bptr, c->status, s);
        }
    } else if (rc == PDB_OK) {
        k_bsp_one_batch<<<1, 1, 0, s>>>(bptr, nnz);
        note_launch();
    }
    if (rc == PDB_OK) {
        k_bsp_gather<<<grid_1d(nnz), 256, 0, s>>>(bpos ? bpos : c->csc_pos, c->col, val, c->row_of, nnz, bcol, brow,
                                                  bval, c->status);
        note_launch();
        k_bsp_runs<<<grid_1d((nnz + 7) / 8), 256, 0, s>>>(skey, bcol, bptr, nnz, runs, n_runs, c->status);
        note_launch();
        if (cudaPeekAtLastError() != cudaSuccess) rc = PDB_ECUDA;
    }
    release(scratch, s);
    return rc;
}

// the two launches of a batch; `follow`: the launch before on this stream is
// this batch's or the batch before's other one, and this kernel may start while
// it drains (launch_next, wait_previous).  `most`: the largest grid (0: any; both
// kernels stride over their work).
struct BspLaunch {
    cudaLaunchConfig_t cfg = {};
    cudaLaunchAttribute attr = {};
    BspLaunch(int64_t blocks, int threads, bool follow, cudaStream_t s)
    {
        cfg.gridDim = dim3((unsigned)blocks);
        cfg.blockDim = dim3((unsigned)threads);
        cfg.stream = s;
        attr.id = cudaLaunchAttributeProgrammaticStreamSerialization;
        attr.val.programmaticStreamSerializationAllowed = 1;
        cfg.attrs = &attr;
        cfg.numAttrs = follow ? 1 : 0;
    }
};
int launch_coef(int64_t r0, int64_t r1, const pdb_csr *X, const float *y, const float *w, int loss, float eta,
                float *coef, const int *status, bool follow, int64_t most, cudaStream_t s)
{
    const int64_t blocks = grid_1d((r1 - r0) * 32);
    const BspLaunch l(most > 0 ? std::min(blocks, most) : blocks, 256, follow, s);
    const cudaError_t e = cudaLaunchKernelEx(&l.cfg, k_bsp_coef, r0, r1, X->row_ptr, X->col, X->val, y, w, loss, eta,
                                             coef, status);
    note_launch();
    return e == cudaSuccess ? PDB_OK : PDB_ECUDA;
}
// pairs: at least the number of the batch's pairs
int launch_apply(int64_t bi, int64_t r0, int64_t rows, int64_t pairs, int sms, const int64_t *bptr, const int32_t *bcol,
                 const int32_t *brow, const float *bval, const int32_t *runs, const uint2 *n_runs, const float *coef,
                 float *w, int *status, bool follow, int64_t most, cudaStream_t s)
{
    // a long run holds more than BSP_LONG pairs, so this covers one block per long run up to the cap
    if (most <= 0) most = (int64_t)sms * BSP_BLOCKS;
    const int64_t blocks = std::max<int64_t>(1, std::min<int64_t>((pairs + BSP_LONG - 1) / BSP_LONG,
                                                                  std::min<int64_t>(most, (int64_t)sms * BSP_BLOCKS)));
    const BspLaunch l(blocks, BSP_THREADS, follow, s);
    const cudaError_t e = cudaLaunchKernelEx(&l.cfg, k_bsp_apply, bi, bptr, (int32_t)r0, (int32_t)rows, bcol, brow,
                                             bval, runs, n_runs, coef, w, status);
    note_launch();
    return e == cudaSuccess ? PDB_OK : PDB_ECUDA;
}

// The grid of k_sgd_ready and the examples a warp takes per ticket.  Two
// examples of k ids conflict with probability ~k^2 / n_cols, so about n_cols /
// k^2 run at once.  Where those are few, a warp's second example per ticket, which
// waits for the first and is loaded only after it, lengthens every chain, and
// warps beyond them only poll; where they are many, the warps cover memory
// latency, and the tickets (one address) bound short rows.  Measured, ms per epoch, 1
// example per ticket with 2 blocks per SM / 2 with 4: 200k examples of 30 ids over 200k
// features (n_cols / k^2 = 222) 1.39 / 3.29; 100k of 60 over 4M (1111) 0.16 / 0.50;
// 500k of 100 over 100M (10000) 2.06 / 2.25 (2.32 at full occupancy); 500k of 30
// over 20M (22222) 0.59 / 0.38.
int ready_grid(const void *kern, const pdb_csr *X, const pdb_opts *opts, int *chunk)
{
    const double k = X->n_rows > 0 ? (double)X->nnz / (double)X->n_rows : 0.0;
    const bool free = (double)X->n_cols > 5000.0 * k * k;
    *chunk = opts && opts->ticket_chunk > 0 ? opts->ticket_chunk : free ? 2 : 1;
    pdb_opts o = opts ? *opts : pdb_opts{};
    if (o.blocks_per_sm <= 0) o.blocks_per_sm = free ? 4 : 2;
    return persistent_grid(kern, &o);
}

int check_run(const pdb_csr *X, const float *y, const pdb_conflicts *c, const float *w, int loss, int epochs)
{
    if (!X || !c || epochs < 0) return PDB_EINVAL;
    if (loss != PDB_LOSS_LOGISTIC && loss != PDB_LOSS_SQUARED && loss != PDB_LOSS_HINGE) return PDB_EINVAL;
    if (X->n_rows != c->n_rows || X->n_cols != c->n_cols || X->nnz != c->nnz) return PDB_EINVAL;
    if (!X->row_ptr || (X->nnz > 0 && !X->col)) return PDB_EINVAL;
    if ((X->n_rows > 0 && !y) || (X->n_cols > 0 && !w)) return PDB_EINVAL;
    return PDB_OK;
}

}  // namespace

extern "C" {

int pdb_sgd_epoch(const pdb_csr *X, const float *y, const pdb_conflicts *c, const pdb_schedule *h, float *w,
                  pdb_loss loss, float eta, int n_epochs, const pdb_opts *opts, void *stream)
{
    ApiScope scope("pdb_sgd_epoch", c, h);
    UseMark use{c, h, (cudaStream_t)stream};
    int rc = check_run(X, y, c, w, loss, n_epochs);
    if (rc != PDB_OK) return rc;
    if (!h || h->c != c) return PDB_EINVAL;
    cudaStream_t s = (cudaStream_t)stream;
    pdb_conflicts *cm = const_cast<pdb_conflicts *>(c);
    const int width = register_width(cm);
    cudaEventRecord(cm->ev_sgd0, s);
    cudaEventRecord(cm->ev_k0, s);
    cudaEventRecord(cm->ev_k1, s);
    const uint64_t tmo = timeout_ns(opts);
    uint64_t *trace = opts ? opts->trace : nullptr;
    int32_t n32 = (int32_t)X->n_rows;
    int lossi = (int)loss;
    if (X->n_rows > 0 && n_epochs > 0) {
        if (h->mode == PDB_SCHED_LEVELS) {
            const void *kern = width == 2 ? (const void *)k_sgd_levels<2>
                               : width == 4 ? (const void *)k_sgd_levels<4> : (const void *)k_sgd_levels<8>;
            int grid = persistent_grid(kern, opts);
            const int64_t *rp = X->row_ptr;
            const int32_t *cl = X->col;
            const float *vl = X->val;
            void *args[] = {(void *)&n32,      (void *)&rp,  (void *)&cl,       (void *)&vl,     (void *)&y,
                            (void *)&h->order, (void *)&h->level_ptr, (void *)&h->ctl, (void *)&w,
                            (void *)&lossi,    (void *)&eta, (void *)&n_epochs, (void *)&h->bar,
                            (void *)&cm->status, (void *)&tmo, (void *)&trace};
            cudaEventRecord(cm->ev_k0, s);
            if (cudaLaunchCooperativeKernel(kern, grid, THREADS, args, 0, s) != cudaSuccess) rc = PDB_ECUDA;
            note_launch();
            cudaEventRecord(cm->ev_k1, s);
        } else if (h->mode == PDB_SCHED_CHAIN) {
            cudaEventRecord(cm->ev_k0, s);
            rc = h->dense ? dense_run(X, y, w, lossi, eta, n_epochs, cm->status, trace, s)
                 : h->resident ? resident_run(X, y, w, lossi, eta, n_epochs, c->h_info[2], cm->status, trace, s)
                             : chain_run(X, y, h->link, w, lossi, eta, n_epochs, c->h_info[2], cm->status, trace, s);
            cudaEventRecord(cm->ev_k1, s);
        } else if (h->mode == PDB_SCHED_WINDOW) {
            cudaEventRecord(cm->ev_k0, s);
            pdb_schedule *hm = const_cast<pdb_schedule *>(h);
            rc = window_run(X, y, c->gate_window, w, h->rec, &hm->epochs_run, h->prog, h->prog_cap, h->wctl, c->near, lossi,
                            eta, n_epochs, width, opts, cm->status, tmo, s);
            cudaEventRecord(cm->ev_k1, s);
        } else if (block_ready_smem(X->n_cols, c->h_info[2]) > 0 && (int64_t)n_epochs * X->n_rows < (1ll << 31) - 1024) {
            // READY with every record in one block's shared memory (few features)
            cudaEventRecord(cm->ev_k0, s);
            rc = block_ready_run(X, y, c->gate, w, lossi, eta, n_epochs, c->h_info[2], cm->status, tmo, trace, s);
            cudaEventRecord(cm->ev_k1, s);
        } else {
            auto kern = width == 2 ? k_sgd_ready<2> : width == 4 ? k_sgd_ready<4> : k_sgd_ready<8>;
            int chunk = 1;
            const int grid = ready_grid((const void *)kern, X, opts, &chunk);
            const int64_t F = X->n_cols;
            k_pack<<<grid_1d(F), 256, 0, s>>>(w, F, h->rec, cm->status);
            note_launch();
            if (fill_words(h->ticket, 0u, sizeof(unsigned long long), s) != PDB_OK) return PDB_ECUDA;
            cudaEventRecord(cm->ev_k0, s);
            kern<<<grid, THREADS, 0, s>>>(n32, X->row_ptr, X->col, X->val, y, c->gate, h->rec, lossi, eta, n_epochs,
                                          h->ticket, chunk, cm->status, tmo, trace);
            note_launch();
            cudaEventRecord(cm->ev_k1, s);
            k_unpack<<<grid_1d(F), 256, 0, s>>>(h->rec, F, w, cm->status);
            note_launch();
        }
    }
    cudaEventRecord(cm->ev_sgd1, s);
    cm->timed_sgd = true;
    if (rc == PDB_OK && cudaPeekAtLastError() != cudaSuccess) rc = PDB_ECUDA;
    if (rc != PDB_OK) cudaGetLastError();
    return rc;
}

int pdb_ssp_epoch(const pdb_csr *X, const float *y, const pdb_conflicts *c, const pdb_schedule *h, float *w,
                  pdb_loss loss, float eta, int n_epochs, int64_t delay, float *coef, const pdb_opts *opts,
                  void *stream)
{
    ApiScope scope("pdb_ssp_epoch", c, h);
    UseMark use{c, h, (cudaStream_t)stream};
    int rc = check_run(X, y, c, w, loss, n_epochs);
    if (rc != PDB_OK) return rc;
    if (!h || h->c != c || delay < 0) return PDB_EINVAL;
    if (h->mode != PDB_SCHED_READY) return PDB_ESTATE;
    const int gates = opts ? opts->ssp_gates : 0;
    if (gates < 0 || gates > PDB_SSP_PREFIX) return PDB_EINVAL;
    const bool prefix = gates == PDB_SSP_PREFIX;
    cudaStream_t s = (cudaStream_t)stream;
    pdb_conflicts *cm = const_cast<pdb_conflicts *>(c);
    pdb_schedule *hm = const_cast<pdb_schedule *>(h);
    const int width = register_width(cm);
    // scratch kept with the schedule, allocated in pairs on first use and
    // attached only when both allocations succeeded
    auto alloc_pair = [&](unsigned **a, unsigned **b, int64_t words) {
        if (*a && *b) return PDB_OK;
        unsigned *x = nullptr, *z = nullptr;
        int r = alloc((void **)&x, sizeof(unsigned) * words, s);
        r = r ? r : alloc((void **)&z, sizeof(unsigned) * words, s);
        if (r != PDB_OK) {
            release(x, s);
            release(z, s);
            return r;
        }
        release(*a, s);
        release(*b, s);
        *a = x;
        *b = z;
        return PDB_OK;
    };
    rc = alloc_pair(&hm->reads, &hm->writes, std::max<int64_t>(X->n_cols, 1));
    if (rc != PDB_OK) return rc;
    // one bit per CSC slot, two words of slack past the last slot's word
    const int64_t n_words = X->nnz / 32 + 2;
    if (prefix) {
        rc = alloc_pair(&hm->rbits, &hm->wbits, n_words);
        if (rc != PDB_OK) return rc;
    }
    cudaEventRecord(cm->ev_sgd0, s);
    cudaEventRecord(cm->ev_k0, s);
    if (X->n_rows > 0 && n_epochs > 0)
        rc = ssp_run(X, y, c->gate, w, hm->writes, hm->reads, h->ticket, (long long)std::min<int64_t>(delay, 1ll << 40),
                     coef, (int)loss, eta, n_epochs, width, opts, cm->status, timeout_ns(opts), s, c->feat_ptr,
                     prefix ? hm->rbits : nullptr, prefix ? hm->wbits : nullptr, n_words);
    cudaEventRecord(cm->ev_k1, s);
    cudaEventRecord(cm->ev_sgd1, s);
    cm->timed_sgd = true;
    if (rc == PDB_OK && cudaPeekAtLastError() != cudaSuccess) rc = PDB_ECUDA;
    if (rc != PDB_OK) cudaGetLastError();
    return rc;
}

int pdb_bsp_epoch(const pdb_csr *X, const float *y, const pdb_conflicts *c, float *w, pdb_loss loss, float eta,
                  int64_t batch, int n_epochs, const pdb_opts *opts, void *stream)
{
    ApiScope scope("pdb_bsp_epoch", c);
    UseMark use{c, nullptr, (cudaStream_t)stream};
    int rc = check_run(X, y, c, w, loss, n_epochs);
    if (rc != PDB_OK) return rc;
    if (batch < 1) return PDB_EINVAL;
    cudaStream_t s = (cudaStream_t)stream;
    pdb_conflicts *cm = const_cast<pdb_conflicts *>(c);
    const int64_t N = X->n_rows, nnz = X->nnz;
    if (batch > N && N > 0) batch = N;
    cudaEventRecord(cm->ev_bsp0, s);
    if (N > 0 && n_epochs > 0) {
        const int64_t n_batches = (N + batch - 1) / batch;
        int32_t *bcol = nullptr, *brow = nullptr;
        float *bval = nullptr, *cbuf = nullptr;
        int64_t *bptr = nullptr;
        int32_t *runs = nullptr;
        uint2 *n_runs = nullptr;
        Block block;
        rc = alloc_block(block, {{(void **)&bcol, sizeof(int32_t) * nnz}, {(void **)&brow, sizeof(int32_t) * nnz},
                                  {(void **)&bval, sizeof(float) * nnz}, {(void **)&cbuf, sizeof(float) * batch},
                                  {(void **)&bptr, sizeof(int64_t) * (n_batches + 1)},
                                  {(void **)&runs, sizeof(int32_t) * nnz},
                                  {(void **)&n_runs, sizeof(uint2) * n_batches}}, s);
        int64_t max_row = 0;
        if (rc == PDB_OK) {
            if (cudaEventSynchronize(c->ev1) != cudaSuccess) {
                cudaGetLastError();
                rc = PDB_ECUDA;
            }
            max_row = c->h_info[2];
        }
        rc = rc ? rc : bsp_sort(cm, X->val, batch, n_batches, bcol, brow, bval, bptr, runs, n_runs, s);
        const int sms = launch_info().sms;
        // blocks_per_sm caps what the call keeps resident: each grid, and no kernel
        // beside the one before it.  Otherwise the first launch waits for everything
        // before it, and the others start early.
        const bool capped = opts && opts->blocks_per_sm > 0;
        const int64_t most = capped ? (int64_t)opts->blocks_per_sm * sms : 0;
        for (int ep = 0; rc == PDB_OK && ep < n_epochs; ++ep)
            for (int64_t b = 0; rc == PDB_OK && b < n_batches; ++b) {
                const int64_t r0 = b * batch, r1 = std::min(N, r0 + batch);
                rc = launch_coef(r0, r1, X, y, w, (int)loss, eta, cbuf, cm->status, !capped && (ep > 0 || b > 0),
                                 most, s);
                if (rc == PDB_OK && nnz > 0)
                    rc = launch_apply(b, r0, r1 - r0, std::min(nnz, (r1 - r0) * max_row), sms, bptr, bcol, brow, bval,
                                      runs, n_runs, cbuf, w, cm->status, !capped, most, s);
            }
        release(block, s);
    }
    cudaEventRecord(cm->ev_bsp1, s);
    cm->timed_bsp = true;
    if (rc == PDB_OK && cudaPeekAtLastError() != cudaSuccess) rc = PDB_ECUDA;
    if (rc != PDB_OK) cudaGetLastError();
    return rc;
}

int pdb_bsp_plan_build(const pdb_conflicts *c, int64_t batch, pdb_bsp_plan **out, void *stream)
{
    ApiScope scope("pdb_bsp_plan_build", c);
    if (!out) return PDB_EINVAL;
    *out = nullptr;
    if (!c || batch < 1) return PDB_EINVAL;
    cudaStream_t s = (cudaStream_t)stream;
    pdb_conflicts *cm = const_cast<pdb_conflicts *>(c);
    const int64_t N = c->n_rows, nnz = c->nnz;
    if (batch > N && N > 0) batch = N;
    pdb_bsp_plan *p = new (std::nothrow) pdb_bsp_plan();
    if (!p) return PDB_ENOMEM;
    p->c = c;
    p->batch = batch;
    if (cudaEventCreateWithFlags(&p->ev_use, cudaEventDisableTiming) != cudaSuccess) {
        cudaGetLastError();
        p->ev_use = nullptr;
    }
    p->n_batches = N > 0 ? (N + batch - 1) / batch : 0;
    int rc = alloc_block(p->arrays, {{(void **)&p->bptr, sizeof(int64_t) * (p->n_batches + 1)},
                                     {(void **)&p->bcol, sizeof(int32_t) * nnz},
                                     {(void **)&p->brow, sizeof(int32_t) * nnz},
                                     {(void **)&p->bval, sizeof(float) * nnz},
                                     {(void **)&p->runs, sizeof(int32_t) * nnz},
                                     {(void **)&p->n_runs, sizeof(uint2) * std::max<int64_t>(p->n_batches, 1)}}, s);
    rc = rc ? rc : bsp_sort(cm, c->val, batch, p->n_batches, p->bcol, p->brow, p->bval, p->bptr, p->runs, p->n_runs, s);
    if (rc == PDB_OK && cudaPeekAtLastError() != cudaSuccess) rc = PDB_ECUDA;
    // the host keeps the batches' pair bounds (apply needs them to size its launch)
    if (rc == PDB_OK) {
        p->h_bptr = new (std::nothrow) int64_t[p->n_batches + 1];
        if (!p->h_bptr) rc = PDB_ENOMEM;
        else if (cudaMemcpyAsync(p->h_bptr, p->bptr, sizeof(int64_t) * (p->n_batches + 1), cudaMemcpyDeviceToHost, s) !=
                     cudaSuccess ||
                 cudaStreamSynchronize(s) != cudaSuccess)
            rc = PDB_ECUDA;
    }
    if (rc != PDB_OK) {
        cudaGetLastError();
        cudaStreamSynchronize(s);
        pdb_bsp_plan_free(p);
        return rc;
    }
    *out = p;
    return PDB_OK;
}

int64_t pdb_bsp_plan_batches(const pdb_bsp_plan *p) { return p ? p->n_batches : -1; }

int pdb_bsp_coef(const pdb_bsp_plan *p, const pdb_csr *X, const float *y, const float *w, pdb_loss loss, float eta,
                 int64_t row_begin, int64_t row_end, float *coef, void *stream)
{
    ApiScope scope("pdb_bsp_coef", p ? p->c : nullptr, nullptr, nullptr, nullptr, false);
    UseMark use{p ? p->c : nullptr, nullptr, (cudaStream_t)stream};
    if (!p) return PDB_EINVAL;
    int rc = check_run(X, y, p->c, w, loss, 1);
    if (rc != PDB_OK) return rc;
    if (row_begin < 0 || row_end < row_begin || row_end > X->n_rows) return PDB_EINVAL;
    if (row_end > row_begin && !coef) return PDB_EINVAL;
    // the rows must lie inside one batch: the margins read that batch's start weights
    if (row_end > row_begin && row_begin / p->batch != (row_end - 1) / p->batch) return PDB_EINVAL;
    if (row_end == row_begin) return PDB_OK;
    cudaStream_t s = (cudaStream_t)stream;
    rc = launch_coef(row_begin, row_end, X, y, w, (int)loss, eta, coef, p->c->status, false, 0, s);
    return rc == PDB_OK && cudaPeekAtLastError() == cudaSuccess ? PDB_OK : PDB_ECUDA;
}

int pdb_bsp_apply(const pdb_bsp_plan *p, float *w, int64_t batch_index, const float *coef, void *stream)
{
    ApiScope scope("pdb_bsp_apply", p ? p->c : nullptr, nullptr, nullptr, nullptr, false);
    UseMark use{p ? p->c : nullptr, nullptr, (cudaStream_t)stream};
    if (!p || batch_index < 0 || batch_index >= p->n_batches) return PDB_EINVAL;
    if (p->c->n_cols > 0 && !w) return PDB_EINVAL;
    const int64_t s0 = p->h_bptr[batch_index], s1 = p->h_bptr[batch_index + 1];
    if (s1 == s0) return PDB_OK;
    if (!coef) return PDB_EINVAL;
    const int64_t r0 = batch_index * p->batch, rows = std::min(p->c->n_rows, r0 + p->batch) - r0;
    cudaStream_t s = (cudaStream_t)stream;
    const int rc = launch_apply(batch_index, r0, rows, s1 - s0, launch_info().sms, p->bptr, p->bcol, p->brow, p->bval,
                                p->runs, p->n_runs, coef, w, const_cast<pdb_conflicts *>(p->c)->status, false, 0, s);
    if (p->ev_use) cudaEventRecord(p->ev_use, s);
    return rc == PDB_OK && cudaPeekAtLastError() == cudaSuccess ? PDB_OK : PDB_ECUDA;
}

void pdb_bsp_plan_free(pdb_bsp_plan *p)
{
    if (!p) return;
    // the plan's own work only: other streams of the device keep running
    if (p->ev_use) {
        cudaEventSynchronize(p->ev_use);
        cudaEventDestroy(p->ev_use);
    }
    cudaGetLastError();
    release(p->arrays, own_stream());
    delete[] p->h_bptr;
    delete p;
}

int pdb_eval_grad(const float *m, const float *y, float *out, int64_t n, pdb_loss loss, void *stream)
{
    if (n < 0 || (n > 0 && (!m || !y || !out))) return PDB_EINVAL;
    if (loss != PDB_LOSS_LOGISTIC && loss != PDB_LOSS_SQUARED && loss != PDB_LOSS_HINGE) return PDB_EINVAL;
    if (n == 0) return PDB_OK;
    k_eval_grad<<<grid_1d(n), 256, 0, (cudaStream_t)stream>>>(m, y, out, n, (int)loss);
    note_launch();
    return cudaPeekAtLastError() == cudaSuccess ? PDB_OK : PDB_ECUDA;
}

int pdb_eval_expf(const float *x, float *out, int64_t n, void *stream)
{
    if (n < 0 || (n > 0 && (!x || !out))) return PDB_EINVAL;
    if (n == 0) return PDB_OK;
    k_eval_expf<<<grid_1d(n), 256, 0, (cudaStream_t)stream>>>(x, out, n); note_launch();
    return cudaPeekAtLastError() == cudaSuccess ? PDB_OK : PDB_ECUDA;
}

}  // extern "C"

// ---------------------------------------------------------------- allocation-free READY epoch
// Some callers cannot let a library allocate device memory while they
// train: a server that has handed all device memory to its own pool and
// must not see it grow or fragment, or a host runtime that accounts for
// every device allocation itself and forbids libraries to make their own.
// For them the READY epoch below keeps its per-feature (weight, version)
// records, its ticket counter and its status word in one fixed array
// compiled into the library instead of in a schedule handle.  Every GPU that
// loads libpdb holds this array (NOALLOC_MAX_COLS * 8 bytes + 256 bytes,
// about 8 MiB) until the process exits.  All calls on a device share it:
// two calls whose work overlaps on the GPU corrupt each other, so order them
// on one stream.
constexpr int64_t NOALLOC_MAX_COLS = 1 << 20;
constexpr int64_t NOALLOC_WORDS = NOALLOC_MAX_COLS + 32;   // records, then ticket and status
static __device__ __align__(256) unsigned long long g_noalloc_scratch[NOALLOC_WORDS];

namespace {

std::mutex g_noalloc_lock;
struct NoallocSlot {
    void *ctx;                  // context the address was looked up in
    unsigned long long *ptr;
};
NoallocSlot g_noalloc_slot[64];

// The driver's current context (nullptr when none is current or the driver
// entry point is unavailable).  A device's module, and with it the scratch
// array, is loaded once per context: after cudaDeviceReset the array may sit
// elsewhere, so the cached address is keyed by context as well as device.
void *current_context()
{
    typedef CUresult (*GetCurrent)(CUcontext *);
    static GetCurrent fn = [] {
        void *f = nullptr;
        cudaDriverEntryPointQueryResult q;
        if (cudaGetDriverEntryPointByVersion("cuCtxGetCurrent", &f, 12000, cudaEnableDefault, &q) != cudaSuccess ||
            q != cudaDriverEntryPointSuccess) {
            cudaGetLastError();
            return (GetCurrent) nullptr;
        }
        return (GetCurrent)f;
    }();
    CUcontext c = nullptr;
    if (!fn || fn(&c) != CUDA_SUCCESS) return nullptr;
    return (void *)c;
}

// Device address of the scratch array for the current device and context.
// Host code only sees a stand-in symbol, not the address, so the address is
// looked up (cudaGetSymbolAddress, with that device current) on the first
// call in each device context and reused afterwards.
unsigned long long *noalloc_scratch()
{
    int dev = 0;
    if (cudaGetDevice(&dev) != cudaSuccess || dev < 0 || dev >= 64) return nullptr;
    std::lock_guard<std::mutex> guard(g_noalloc_lock);
    NoallocSlot &slot = g_noalloc_slot[dev];
    void *ctx = current_context();
    if (!slot.ptr || !ctx || ctx != slot.ctx) {
        void *p = nullptr;
        if (cudaGetSymbolAddress(&p, g_noalloc_scratch) != cudaSuccess) {
            cudaGetLastError();
            slot.ptr = nullptr;
            return nullptr;
        }
        slot.ptr = (unsigned long long *)p;
        slot.ctx = current_context();   // the lookup makes the device's primary context current
    }
    return slot.ptr;
}

}  // namespace

extern "C" int pdb_sgd_epoch_ready_noalloc(const pdb_csr *X, const float *y, const uint32_t *gate, float *w,
                                           pdb_loss loss, float eta, int n_epochs, void *stream)
{
    ApiScope scope("pdb_sgd_epoch_ready_noalloc", nullptr, nullptr, nullptr, nullptr, false);  // no handle to log
    if (!X || X->n_rows < 0 || X->n_cols < 0 || X->nnz < 0 || n_epochs < 0) return PDB_EINVAL;
    if (X->n_cols > NOALLOC_MAX_COLS) return PDB_ETOOBIG;
    if (X->n_rows >= (1ll << 31) - 1 || X->nnz >= (1ll << 31) - 1) return PDB_EINVAL;
    if (loss != PDB_LOSS_LOGISTIC && loss != PDB_LOSS_SQUARED && loss != PDB_LOSS_HINGE) return PDB_EINVAL;
    if (!X->row_ptr || (X->nnz > 0 && (!X->col || !gate)) || (X->n_rows > 0 && !y) || (X->n_cols > 0 && !w))
        return PDB_EINVAL;
    unsigned long long *scratch = noalloc_scratch();
    if (!scratch) return PDB_ECUDA;
    unsigned long long *rec = scratch;
    unsigned long long *ticket = scratch + NOALLOC_MAX_COLS;
    int *status = (int *)(scratch + NOALLOC_MAX_COLS + 1);
    cudaStream_t s = (cudaStream_t)stream;
    // the previous call left its status and ticket behind: start from zero
    if (fill_words(status, 0u, sizeof(int), s) != PDB_OK) return PDB_ECUDA;
    if (X->n_rows > 0 && n_epochs > 0) {
        const int64_t F = X->n_cols;
        const int32_t n32 = (int32_t)X->n_rows;
        const uint64_t tmo = timeout_ns(nullptr);
        int chunk = 1;
        const int grid = ready_grid((const void *)k_sgd_ready<8>, X, nullptr, &chunk);
        if (F > 0) {
            k_pack<<<grid_1d(F), 256, 0, s>>>(w, F, rec, status);
            note_launch();
        }
        if (fill_words(ticket, 0u, sizeof(unsigned long long), s) != PDB_OK) return PDB_ECUDA;
        k_sgd_ready<8><<<grid, THREADS, 0, s>>>(n32, X->row_ptr, X->col, X->val, y, gate, rec, (int)loss, eta,
                                                n_epochs, ticket, chunk, status, tmo, nullptr);
        note_launch();
        if (F > 0) {
            k_unpack<<<grid_1d(F), 256, 0, s>>>(rec, F, w, status);
            note_launch();
        }
    }
    if (cudaPeekAtLastError() != cudaSuccess) {
        cudaGetLastError();
        return PDB_ECUDA;
    }
    int st = 0;
    if (cudaMemcpyAsync(&st, status, sizeof(int), cudaMemcpyDeviceToHost, s) != cudaSuccess ||
        cudaStreamSynchronize(s) != cudaSuccess)
        return PDB_ECUDA;
    return st;
}
