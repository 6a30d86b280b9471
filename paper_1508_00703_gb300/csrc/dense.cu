// Dense chain engine: pdb_sgd_epoch under a CHAIN schedule when every example
// holds every feature, ids in order (row t is val[t F .. (t + 1) F)), and the
// F weights fit one warp's registers.
//
// Every example then reads and writes the same F weights, so the examples run
// one after the other (Algorithm 1 itself), and lane l can keep the weights of
// the features l, l + 32, ... in registers for the whole call: an example needs
// its values only, no ids, no weight loads or stores.
//
//   compute   one warp: per element the step of the example before (w = w - c x,
//             two roundings) directly followed by this example's fused
//             multiply-add (the fp32 operations and order of every engine),
//             then the combine and the derivative;
//   copy      8 warps, one example of a step of 8 each: values from global
//             memory into registers in one step, from there into a
//             shared-memory ring in the next (any row alignment).
//
// What bounds it: the chain of F / 32 dependent multiply-adds per lane (4
// cycles each), the two-round combine (~85 cycles) and the derivative, of one
// example after the other; the three instructions per element fit in the
// multiply-add's latency.  In the ring, a lane's values are neighbours (one
// 16-byte load per four; rows of R + 4 words per lane spread them over the
// banks).  The resident-weight engine ran the same data with ids, values and
// weights from shared memory, 90 loads per lane and example.  Measured, 960
// features, squared loss: 618 -> 145 ns per example (~290 cycles; alone, with
// nothing to copy, 271: 115 the multiply-adds, ~125 combine and derivative).
#include <cuda_runtime.h>

#include <atomic>

#include "common.cuh"

using namespace pdb;

namespace {

constexpr int DN_G = 8;                 // examples per step
constexpr int DN_RING = 4;              // steps in the ring: being read, read ahead, being written (power of two)
constexpr int DN_THREADS = 384;         // warp 0 computes, alone on its scheduler with warps 4 and 8, which only wait
constexpr int DN_MAX = 1024;            // most features (32 per lane)

template <int R>
struct DenseSmem {
    float x[DN_RING * DN_G][32][R + 4]; // element q * 32 + l of an example at [l][q]
    float y[DN_RING * DN_G];
};

template <int R>
__device__ __forceinline__ void load_values(const DenseSmem<R> &S, int slot, int lane, float (&x)[R])
{
#pragma unroll
    for (int q = 0; q < R; q += 4) {
        const float4 v = *reinterpret_cast<const float4 *>(&S.x[slot][lane][q]);
        x[q] = v.x;
        x[q + 1] = v.y;
        x[q + 2] = v.z;
        x[q + 3] = v.w;
    }
}

// w -= c * xp; the elements past F keep weight +0 (values there are -0: their
// products leave a partial sum as it is), also when c is not finite.  R is F /
// 32 rounded up to a multiple of 4, so only the last four can be past it.
template <int R>
__device__ __forceinline__ float step_weight(float w, float c, float xp, int q, int lane, int F)
{
    const float n = __fsub_rn(w, __fmul_rn(c, xp));
    return q < R - 4 || q * 32 + lane < F ? n : 0.0f;
}

// One example: the step c of the example before (values xp) and the margin in
// one sweep over the elements, xp taking the next example's values behind it.
// Returns this example's step.
template <int R, int LOSS, bool TRACE>
__device__ __forceinline__ float dense_example(const DenseSmem<R> &S, float (&w)[R], float (&xp)[R], const float (&x)[R],
                                               float c, int slot, int next, int lane, int F, float eta, uint64_t *trace,
                                               int64_t idx)
{
    const float y = S.y[slot];
    float a = 0.0f;
#pragma unroll
    for (int q = 0; q < R; q += 4) {
#pragma unroll
        for (int e = 0; e < 4; ++e) {
            w[q + e] = step_weight<R>(w[q + e], c, xp[q + e], q + e, lane, F);
            a = __fmaf_rn(w[q + e], x[q + e], a);
        }
        const float4 v = *reinterpret_cast<const float4 *>(&S.x[next][lane][q]);
        xp[q] = v.x;
        xp[q + 1] = v.y;
        xp[q + 2] = v.z;
        xp[q + 3] = v.w;
    }
    if (TRACE) trace_mark(trace, idx, 0);
    const float m = warp_combine_latency(a);
    bool general = false;
    float s = dev_step_fast(LOSS, m, y, eta, general);
    if (LOSS == PDB_LOSS_LOGISTIC && general) s = __fmul_rn(eta, dev_grad(LOSS, m, y));
    if (TRACE) trace_mark(trace, idx, 1);   // before any write is visible
    return s;
}

template <int R, int LOSS, bool TRACE>
__global__ __launch_bounds__(DN_THREADS, 1) void k_sgd_dense(int32_t n_rows, int F, const float *__restrict__ val,
                                                             const float *__restrict__ y, float *w_out, float eta,
                                                             int epochs, const int *status, uint64_t *trace)
{
    extern __shared__ __align__(16) unsigned char smem_raw[];
    DenseSmem<R> &S = *reinterpret_cast<DenseSmem<R> *>(smem_raw);
    if (read_status(status)) return;
    constexpr int SLOTS = DN_RING * DN_G;
    const int lane = threadIdx.x & 31, warp = threadIdx.x >> 5;
    const int copier = (warp & 3) ? warp - 1 - (warp >> 2) : -1;     // 0..8 on schedulers 1-3
    const int64_t total = (int64_t)epochs * n_rows;                  // examples of all epochs, in order
    const int64_t steps = (total + DN_G - 1) / DN_G;
    // iteration t: compute step t; write step t + 2's values to the ring; load step t + 3's
    if (warp == 0) {
        float w[R], xa[R], xb[R], c = 0.0f;      // xa, xb: values of the example before and of this one, in turn
#pragma unroll
        for (int q = 0; q < R; ++q) {
            w[q] = q * 32 + lane < F ? w_out[q * 32 + lane] : 0.0f;
            xa[q] = 0.0f;                         // the first example has no step before it: w - 0 * 0
        }
        for (int64_t t = -3; t < steps; ++t) {
            if (t >= 0) {
                const int s0 = (int)((t * DN_G) & (SLOTS - 1)), nx = (s0 + DN_G) & (SLOTS - 1);
                const int n = (int)min64(DN_G, total - t * DN_G);
                const int64_t idx = t * DN_G;
                if (t == 0) load_values(S, 0, lane, xb);
                if (n == DN_G) {
#pragma unroll
                    for (int g = 0; g < DN_G; g += 2) {
                        c = dense_example<R, LOSS, TRACE>(S, w, xa, xb, c, s0 + g, s0 + g + 1, lane, F, eta, trace, idx + g);
                        c = dense_example<R, LOSS, TRACE>(S, w, xb, xa, c, s0 + g + 1, g + 2 < DN_G ? s0 + g + 2 : nx, lane, F,
                                                   eta, trace, idx + g + 1);
                    }
                } else {
#pragma unroll 1
                    for (int g = 0; g < n; ++g) {
                        c = dense_example<R, LOSS, TRACE>(S, w, xa, xb, c, s0 + g, (s0 + g + 1) & (SLOTS - 1), lane, F, eta,
                                                   trace, idx + g);
#pragma unroll
                        for (int q = 0; q < R; ++q) {
                            const float v = xa[q];
                            xa[q] = xb[q];
                            xb[q] = v;
                        }
                    }
                }
            }
            __syncthreads();
        }
        // the last example's step (its values are in xa)
#pragma unroll
        for (int q = 0; q < R; ++q)
            if (q * 32 + lane < F) w_out[q * 32 + lane] = total > 0 ? __fsub_rn(w[q], __fmul_rn(c, xa[q])) : w[q];
    } else {
        float v[R], yv = 0.0f;
#pragma unroll
        for (int q = 0; q < R; ++q) v[q] = -0.0f;
        for (int64_t t = -3; t < steps; ++t) {
            if (copier >= 0 && copier < DN_G) {
                const int64_t rw = (t + 2) * DN_G + copier, rl = (t + 3) * DN_G + copier;
                if (rw >= 0 && rw < total) {
                    const int slot = (int)(rw & (SLOTS - 1));
#pragma unroll
                    for (int q = 0; q < R; q += 4)
                        *reinterpret_cast<float4 *>(&S.x[slot][lane][q]) = make_float4(v[q], v[q + 1], v[q + 2], v[q + 3]);
                    if (lane == 0) S.y[slot] = yv;
                }
                if (rl >= 0 && rl < total) {
                    const int64_t r = rl % n_rows;
                    const float *p = val + r * F + lane;
                    yv = y[r];
#pragma unroll
                    for (int q = 0; q < R; ++q)
                        if (q * 32 + lane < F) v[q] = val ? __ldcs(p + q * 32) : 1.0f;
                }
            }
            __syncthreads();
        }
    }
}

using DenseKernel = void (*)(int32_t, int, const float *, const float *, float *, float, int, const int *, uint64_t *);
struct DenseVariant {
    DenseKernel kern;
    size_t smem;
};
template <int R, bool TRACE>
DenseVariant dense_variant(int loss)
{
    return {loss == PDB_LOSS_LOGISTIC ? k_sgd_dense<R, PDB_LOSS_LOGISTIC, TRACE>
            : loss == PDB_LOSS_SQUARED ? k_sgd_dense<R, PDB_LOSS_SQUARED, TRACE>
                                       : k_sgd_dense<R, PDB_LOSS_HINGE, TRACE>,
            sizeof(DenseSmem<R>)};
}

// weights per lane: 4, 8, .. 32
template <bool TRACE>
DenseVariant dense_variant(int variant, int loss)
{
    switch (variant) {
    case 0: return dense_variant<4, TRACE>(loss);
    case 1: return dense_variant<8, TRACE>(loss);
    case 2: return dense_variant<12, TRACE>(loss);
    case 3: return dense_variant<16, TRACE>(loss);
    case 4: return dense_variant<20, TRACE>(loss);
    case 5: return dense_variant<24, TRACE>(loss);
    case 6: return dense_variant<28, TRACE>(loss);
    default: return dense_variant<32, TRACE>(loss);
    }
}

}  // namespace

namespace pdb {

// Whether this engine takes the data: every row holds all n_cols ids in
// ascending order.  Rows are at most max_row ids and together nnz, so with
// nnz = n_rows n_cols and max_row = n_cols each holds n_cols; ids in range and
// strictly ascending (no descent inside a row) are then 0 .. n_cols - 1.
bool dense_fits(int64_t n_rows, int64_t n_cols, int64_t nnz, int64_t max_row, bool ascending)
{
    return ascending && n_cols >= 1 && n_cols <= DN_MAX && max_row == n_cols && nnz == n_rows * n_cols;
}

int dense_run(const pdb_csr *X, const float *y, float *w, int loss, float eta, int epochs, const int *status,
              uint64_t *trace, cudaStream_t s)
{
    // one kernel per register count, loss and whether it stamps an execution trace
    const int variant = (int)((X->n_cols + 127) / 128) - 1;
    const DenseVariant v = trace ? dense_variant<true>(variant, loss) : dense_variant<false>(variant, loss);
    // set once per device and variant (any device past the table: every call)
    static std::atomic<bool> configured[64][48];
    int dev = 0;
    cudaGetDevice(&dev);
    const bool known = dev >= 0 && dev < 64;
    const int slot = (variant * 3 + (loss >= 0 && loss <= 2 ? loss : 2)) * 2 + (trace ? 1 : 0);
    if (!known || !configured[dev][slot].load(std::memory_order_acquire)) {
        if (cudaFuncSetAttribute((const void *)v.kern, cudaFuncAttributeMaxDynamicSharedMemorySize, (int)v.smem) !=
            cudaSuccess)
            return PDB_ECUDA;
        if (known) configured[dev][slot].store(true, std::memory_order_release);
    }
    v.kern<<<1, DN_THREADS, v.smem, s>>>((int32_t)X->n_rows, (int)X->n_cols, X->val, y, w, eta, epochs, status, trace);
    note_launch();
    return cudaPeekAtLastError() == cudaSuccess ? PDB_OK : PDB_ECUDA;
}

}  // namespace pdb
