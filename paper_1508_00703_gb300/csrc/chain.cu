// Chain engine: pdb_sgd_epoch under a CHAIN schedule.
//
// When the conflict graph is close to one chain (a feature present in most
// examples makes every example depend on the one before), the concurrency
// the read and write constraints allow (Theorem 2) is about one example at a
// time, and what bounds the run is the latency of one dependency hop.  Here
// one thread block runs the examples strictly in data order -- the
// sequential computation of Algorithm 1 itself -- so a hop costs a few
// hundred cycles instead of a round trip through L2:
//
//   compute    one warp runs example after example (the fp32 operations and
//              order of the other engines), and stores each new weight whose
//              next occurrence lies in one of the next D examples straight
//              into that example's weight slot in shared memory;
//   prefetch   G warps, one example of a step each: row bounds, then ids,
//              values, link words and label, then the weights nobody will
//              push, each one step after the one before and held in
//              registers in between (the loads' latency is a step);
//   write      warps that store the new weights of the previous step that are
//              not pushed through to global memory.
//
// A pipeline step handles G consecutive examples, so the fixed cost of a step
// (one barrier, ~180 cycles) is shared by G hops.
//
// What bounds it: the compute warp's chain through one example -- store of the
// example before to shared memory, load, fused multiply-adds, combine,
// derivative (~230 cycles alone for 20 logistic ids, of which the derivative
// ~80, the combine ~55, the store and load ~40).  The helpers finish their step
// first.  Kept short by: one warp for the whole chain (two taking the examples
// in turn spent ~100 cycles per hop on handing over), the derivative without a
// branch (a branch, taken or not, costs ~50 cycles per example: the rare
// margins outside its range are flagged and their step run again), the step's
// examples unrolled (a loop branch costs ~25), loads of everything but the
// weights one example ahead or behind the weights' loads, and helpers that hold
// their loads in registers for a step (asynchronous copies of single elements
// cost 36-80 cycles of issue each).  Measured, ns per example, before and
// after: 20 ids zipf(1.0), logistic 193 -> 118; 50 binary ids zipf(1.1),
// logistic 273 -> 137; 200 ids zipf(1.3), hinge 343 -> 167 (all with this
// engine as the only work on the GPU, the build included in neither).
//
// Ordering: a pushed weight (next occurrence within D examples) is written by
// the compute warp before it computes the consumer (program order); a
// gathered weight's last writer lies more than D examples back, so its
// global store was issued at least one step before the gather, with
// __syncthreads between.  The pipeline drains at every epoch boundary.  No
// spin waits.
#include <cuda_runtime.h>

#include <atomic>
#include <cstddef>

#include "common.cuh"

using namespace pdb;

namespace {

// Pipeline shape for rows of up to 32 R ids.  G examples per step; a step's
// row bounds are loaded RS steps before its compute, its ids AS steps, its
// weights BS steps before; D = G * DS the forwarding window (examples).  Each
// array is a ring of as many example slots as its entries' life needs: values
// and store addresses XS, weights and write-through ids WS, new weights on
// their way out OS (so rows of 256 ids keep 8 examples per step in shared
// memory).  WPER examples per write-through warp.
template <int R>
struct ChainCfg {
    static constexpr int G = 8;
    static constexpr int DS = 5;
    static constexpr int BS = 3, AS = BS + 1, RS = AS + 1;
    static constexpr int PS = RS + 4;               // steps between a row's L2 prefetch and its compute
    static constexpr int D = G * DS;
    static constexpr int XS = 32, WS = 64, OS = 16;
    static constexpr int MAXK = 32 * R;             // longest example
    static constexpr int WPER = 2;
    static constexpr int THREADS = 512;
};
constexpr int CH_MAXK = 256;                        // longest example this engine takes
// link word of a position: bit 31 = its weight will be pushed by an earlier
// example (skip the gather); bit 30 = push the new weight to the next
// occurrence, which is element (bits 0..7) of the example (bits 16..23)
// examples later
constexpr uint32_t LK_RECV = 1u << 31, LK_PUSH = 1u << 30;
template <int R>
constexpr bool chain_cfg_ok()
{
    using C = ChainCfg<R>;
    return (C::XS & (C::XS - 1)) == 0 && (C::WS & (C::WS - 1)) == 0 && (C::OS & (C::OS - 1)) == 0 &&
           C::XS % C::G == 0 && C::WS % C::G == 0 && C::OS % C::G == 0 &&   // a step's slots are neighbours
           // lives, in steps around a step s: values and store addresses s - BS .. s; weights
           // (pushed from s - DS on) s - DS .. s and ids s - BS .. s + 1; out s .. s + 1
           C::XS >= (C::BS + 1) * C::G && C::WS >= (C::DS + 1) * C::G && C::WS >= (C::BS + 2) * C::G &&
           C::OS >= 2 * C::G && C::DS >= C::BS &&
           C::D < 256 && C::MAXK <= 256 &&                                // link word fields
           (C::G & (C::G - 1)) == 0 && C::G <= 8 &&
           // a weight is gathered (not pushed) when its last writer r' lies more
           // than D examples back; r' stores it through at step r'/G + 1, the gather
           // for r runs at step r/G - BS, and r/G - r'/G >= (D + 1) / G: the store
           // lands at least one step (one __syncthreads) before the gather
           (C::D + 1) / C::G >= C::BS + 2 &&
           // the weights gathered for a step are stored to its slots BS - 1 steps
           // before its compute, its values BS steps before: both are in place when
           // the compute warp loads the values of the step's first example, one step
           // before its compute
           C::BS >= 2;
}

static_assert(ChainCfg<8>::MAXK == CH_MAXK, "longest example");

// Layout of the arrays the compute warp reads (xa, pa, wp): element i of an
// example adds into partial sum i mod 32.  Rows of up to 64 ids: the compute
// warp keeps the four partials p, p + 8, p + 16, p + 24 in one lane (the four
// groups of 8 lanes sum the same ones), so those four elements of each 32 are
// neighbours, one 16-byte load; that saves two of the combine's five exchange
// levels.  Longer rows keep one partial per lane: four times fewer loads,
// which is what bounds them.  Elements past the example's end hold value -0
// and weight +0: their product -0 leaves any partial as it is.
template <int R>
constexpr bool QUAD = R <= 2;
template <int R>
__host__ __device__ constexpr int chain_at(int i)
{
    return QUAD<R> ? (i & ~31) | ((i & 7) << 2) | ((i >> 3) & 3) : i;
}

template <int R>
struct ChainSmem {
    using C = ChainCfg<R>;
    // element i at chain_at<R>(i)
    float xa[C::XS][C::MAXK];       // value of each element (1 without values)
    uint32_t pa[C::XS][C::MAXK];    // shared-memory address of each element's new weight
    float wp[C::WS][C::MAXK];       // weight each element reads (gathered or pushed)
    // element i at i
    float out[C::OS][C::MAXK];      // new weight of the elements whose next occurrence is not pushed
    int32_t wcol[C::WS][C::MAXK];   // their ids, -1 for every other element
    float y[C::XS];
    float dump[32];                 // store target of the elements past an example's end
};

// Roles of the warps (scheduler = warp index mod 4): warp 0 computes, alone
// on its scheduler (the other warps there only join the barriers, so nothing
// else issues or fetches instructions beside it); of the warps of schedulers
// 1-3, in index order, the first G prefetch one example g of a step each and
// the next ones write WPER examples' weights through each.
enum { ROLE_PREFETCH, ROLE_WRITE };
// the (first) example of a step that warp serves in the given role, -1 for none
template <int R>
__host__ __device__ constexpr int chain_role(int warp, int kind)
{
    using C = ChainCfg<R>;
    const int role = (warp & 3) ? warp - 1 - (warp >> 2) : -1;
    if (kind == ROLE_PREFETCH) return role >= 0 && role < C::G ? role : -1;
    return role >= C::G && role < C::G + C::G / C::WPER ? C::WPER * (role - C::G) : -1;
}

// every role taken by exactly one warp, none of them the compute warp
template <int R>
constexpr bool chain_roles_ok()
{
    using C = ChainCfg<R>;
    int seen[2] = {0, 0}, writes = 0;
    for (int warp = 0; warp < C::THREADS / 32; ++warp)
        for (int kind = 0; kind < 2; ++kind) {
            const int g = chain_role<R>(warp, kind);
            if (g < 0) continue;
            if (warp % 4 == 0 || g >= C::G || (seen[kind] >> g) & 1 || chain_role<R>(warp, 1 - kind) >= 0) return false;
            seen[kind] |= 1 << g;
        }
    for (int g = 0; g < C::G; g += C::WPER) writes |= 1 << g;
    return seen[ROLE_PREFETCH] == (1 << C::G) - 1 && seen[ROLE_WRITE] == writes;
}
template <int R>
constexpr bool chain_ok()
{
    static_assert(chain_cfg_ok<R>() && chain_roles_ok<R>() && sizeof(ChainSmem<R>) <= 227 * 1024, "chain pipeline shape");
    return true;
}
static_assert(chain_ok<1>() && chain_ok<2>() && chain_ok<3>() && chain_ok<4>() && chain_ok<5>() && chain_ok<6>() &&
              chain_ok<7>() && chain_ok<8>(), "every row width");

__device__ __forceinline__ void st_shared(unsigned addr, float v)
{
    asm volatile("st.shared.f32 [%0], %1;" ::"r"(addr), "f"(v) : "memory");
}
__device__ __forceinline__ float4 ld_shared4(unsigned addr)
{
    float4 v;
    asm volatile("ld.shared.v4.f32 {%0, %1, %2, %3}, [%4];"
                 : "=f"(v.x), "=f"(v.y), "=f"(v.z), "=f"(v.w)
                 : "r"(addr)
                 : "memory");
    return v;
}
__device__ __forceinline__ float ld_shared(unsigned addr)
{
    float v;
    asm volatile("ld.shared.f32 %0, [%1];" : "=f"(v) : "r"(addr) : "memory");
    return v;
}
// *p when `on`, else 0 without an access
__device__ __forceinline__ float ld_if(const float *p, bool on)
{
    float v;
    asm volatile("{\n\t.reg .pred p;\n\tsetp.ne.s32 p, %2, 0;\n\tmov.f32 %0, 0f00000000;\n\t@p ld.global.cg.f32 %0, [%1];\n\t}"
                 : "=f"(v)
                 : "l"(p), "r"((int)on)
                 : "memory");
    return v;
}
__device__ __forceinline__ void prefetch_l2(const void *p) { asm volatile("prefetch.global.L2 [%0];" ::"l"(p)); }

// The upper two levels of the combine tree (partials 16 and 8 apart) add
// within the lane that holds four partials; the lower three (4, 2, 1) take one
// round of seven independent shuffles instead of three dependent ones: lane l
// adds the leaves of its partners' subtrees itself.  Every addition has the
// operands of warp_combine's (fp32 addition commutes), so the same bits.
__device__ __forceinline__ float combine4(float a0, float a1, float a2, float a3)
{
    const float s = __fadd_rn(__fadd_rn(a0, a2), __fadd_rn(a1, a3));
    const float b4 = __shfl_xor_sync(FULL, s, 4), b2 = __shfl_xor_sync(FULL, s, 2), b6 = __shfl_xor_sync(FULL, s, 6);
    const float b1 = __shfl_xor_sync(FULL, s, 1), b5 = __shfl_xor_sync(FULL, s, 5);
    const float b3 = __shfl_xor_sync(FULL, s, 3), b7 = __shfl_xor_sync(FULL, s, 7);
    return __fadd_rn(__fadd_rn(__fadd_rn(s, b4), __fadd_rn(b2, b6)),
                     __fadd_rn(__fadd_rn(b1, b5), __fadd_rn(b3, b7)));
}

// What the compute warp carries from example to example.
template <int R>
struct ChainWarp {
    int lane, at4;          // at4 (QUAD): this lane's four neighbouring elements of each 32
    unsigned base;          // of the block's ChainSmem
    float x[QUAD<R> ? 4 * R : R];   // values of the next example's elements
    bool redo;              // a margin outside dev_step_fast's range
};

// an array's elements that this lane sums, from the row at shared-memory address `row`
template <int R>
__device__ __forceinline__ void load_sum(unsigned row, const ChainWarp<R> &cw, float *v)
{
#pragma unroll
    for (int q = 0; q < R; ++q)
        if (QUAD<R>) {
            const float4 f = ld_shared4(row + 4u * (unsigned)(q * 32 + cw.at4));
            v[4 * q] = f.x;
            v[4 * q + 1] = f.y;
            v[4 * q + 2] = f.z;
            v[4 * q + 3] = f.w;
        } else {
            v[q] = ld_shared(row + 4u * (unsigned)(q * 32 + cw.lane));
        }
}

// One example: weights from its slot (all in place once the example before
// has stored its new ones), margin, step, new weights to their next readers'
// slots or to out.  Values are loaded one example ahead (nslot of xa).  Every other
// load of the example is issued behind its weights' loads, in their latency.
template <int R, int LOSS, bool TRACE, bool FAST>
__device__ __forceinline__ void chain_example(ChainWarp<R> &cw, int wslot, int xslot, int nslot, float eta,
                                              uint64_t *trace, int64_t idx)
{
    using S = ChainSmem<R>;
    constexpr int NS = QUAD<R> ? 4 * R : R;
    const unsigned wrow = 4u * (unsigned)(wslot * ChainCfg<R>::MAXK), xrow = 4u * (unsigned)(xslot * ChainCfg<R>::MAXK);
    // of each 32, the element this lane updates: lane (at chain_at(lane))
    const unsigned own = 4u * (unsigned)(QUAD<R> ? cw.at4 + (cw.lane >> 3) : cw.lane);
    float w[NS], xn[NS], wo[R], xo[R], m;
    unsigned pa[R];
    load_sum<R>(cw.base + (unsigned)offsetof(S, wp) + wrow, cw, w);
    const float y = ld_shared(cw.base + (unsigned)offsetof(S, y) + 4u * (unsigned)xslot);
#pragma unroll
    for (int q = 0; q < R; ++q) {
        if (QUAD<R>) {
            wo[q] = ld_shared(cw.base + (unsigned)offsetof(S, wp) + wrow + 128u * q + own);
            xo[q] = ld_shared(cw.base + (unsigned)offsetof(S, xa) + xrow + 128u * q + own);
        } else {
            wo[q] = w[q];
            xo[q] = cw.x[q];
        }
        pa[q] = __float_as_uint(ld_shared(cw.base + (unsigned)offsetof(S, pa) + xrow + 128u * q + own));
    }
    load_sum<R>(cw.base + (unsigned)offsetof(S, xa) + 4u * (unsigned)(nslot * ChainCfg<R>::MAXK), cw, xn);
    if (QUAD<R>) {
        float a[4] = {0.0f, 0.0f, 0.0f, 0.0f};
#pragma unroll
        for (int q = 0; q < R; ++q)
#pragma unroll
            for (int e = 0; e < 4; ++e) a[e] = __fmaf_rn(w[4 * q + e], cw.x[4 * q + e], a[e]);
        if (TRACE) trace_mark(trace, idx, 0);    // every weight is read
        m = combine4(a[0], a[1], a[2], a[3]);
    } else {
        float a = 0.0f;
#pragma unroll
        for (int q = 0; q < R; ++q) a = __fmaf_rn(w[q], cw.x[q], a);
        if (TRACE) trace_mark(trace, idx, 0);    // every weight is read
        m = warp_combine_latency(a);
    }
    const float c = FAST ? dev_step_fast(LOSS, m, y, eta, cw.redo) : __fmul_rn(eta, dev_grad(LOSS, m, y));
    if (TRACE) trace_mark(trace, idx, 1);    // before any write is visible
#pragma unroll
    for (int q = 0; q < R; ++q) st_shared(pa[q], __fsub_rn(wo[q], __fmul_rn(c, xo[q])));
    __syncwarp();
#pragma unroll
    for (int q = 0; q < NS; ++q) cw.x[q] = xn[q];
}

template <int R, int LOSS, bool TRACE>
__global__ __launch_bounds__(ChainCfg<R>::THREADS, 1) void k_sgd_chain(int32_t n_rows, const int64_t *__restrict__ row_ptr,
                                                             const int32_t *__restrict__ col,
                                                             const float *__restrict__ val,
                                                             const float *__restrict__ y,
                                                             const uint32_t *__restrict__ link, float *w,
                                                             float eta, int epochs, int *status, uint64_t *trace)
{
    using C = ChainCfg<R>;
    extern __shared__ __align__(16) unsigned char smem_raw[];
    ChainSmem<R> &S = *reinterpret_cast<ChainSmem<R> *>(smem_raw);
    if (read_status(status)) return;
    const int lane = threadIdx.x & 31, warp = threadIdx.x >> 5;
    const int gP = chain_role<R>(warp, ROLE_PREFETCH), gW = chain_role<R>(warp, ROLE_WRITE);
    const int N = n_rows;
    const int steps = (N + C::G - 1) / C::G;
    const unsigned wp_base = (unsigned)__cvta_generic_to_shared(&S.wp[0][0]);
    if (warp == 0) {
        ChainWarp<R> cw;
        cw.lane = lane;
        cw.at4 = (lane & 7) * 4;
        cw.base = (unsigned)__cvta_generic_to_shared(smem_raw);
        for (int ep = 0; ep < epochs; ++ep)
            for (int t = -C::PS; t <= steps; ++t) {
                if (t >= 0 && t < steps) {
                    const int r0 = t * C::G, w0 = r0 & (C::WS - 1), x0 = r0 & (C::XS - 1), n = min(N - r0, C::G);
                    const int nx = (x0 + C::G) & (C::XS - 1);   // the next step's first example
                    const int64_t idx = (int64_t)ep * N + r0;
                    if (t == 0) load_sum<R>(cw.base + (unsigned)offsetof(ChainSmem<R>, xa) + 4u * (unsigned)(x0 * C::MAXK), cw, cw.x);
                    cw.redo = false;
                    if (n == C::G) {
#pragma unroll
                        for (int g = 0; g < C::G; ++g)
                            chain_example<R, LOSS, TRACE, true>(cw, w0 + g, x0 + g, g + 1 < C::G ? x0 + g + 1 : nx, eta,
                                                                trace, idx + g);
                    } else {
#pragma unroll 1
                        for (int g = 0; g < n; ++g)
                            chain_example<R, LOSS, TRACE, true>(cw, w0 + g, x0 + g, (x0 + g + 1) & (C::XS - 1), eta,
                                                                trace, idx + g);
                    }
                    if (cw.redo) {
                        // the whole step again with the general derivative: its examples'
                        // own slots hold what they read (a step's stores go to later
                        // examples), and every store of the first run is made again
                        load_sum<R>(cw.base + (unsigned)offsetof(ChainSmem<R>, xa) + 4u * (unsigned)(x0 * C::MAXK), cw, cw.x);
#pragma unroll 1
                        for (int g = 0; g < n; ++g)
                            chain_example<R, LOSS, TRACE, false>(cw, w0 + g, x0 + g, (x0 + g + 1) & (C::XS - 1), eta,
                                                                 trace, idx + g);
                    }
                }
                __syncthreads();
            }
    } else if (gP >= 0) {
        const unsigned out_base = (unsigned)__cvta_generic_to_shared(&S.out[0][0]);
        const unsigned dump = (unsigned)__cvta_generic_to_shared(&S.dump[lane]);
        for (int ep = 0; ep < epochs; ++ep) {
            int32_t cc[R];              // ids, link words, values and label of step t + AS
            uint32_t lk[R];
            float xv[R], yv = 0.0f, wg[R];
            unsigned recv = ~0u;        // elements whose slot takes a pushed weight, not wg
            int64_t b = 0, e = 0;       // row bounds of step t + RS
            int64_t pb = 0, pe = 0;     // row bounds of step t + PS
            int k = 0;                  // row length of step t + AS
#pragma unroll
            for (int q = 0; q < R; ++q) {
                cc[q] = 0;
                lk[q] = 0u;
                xv[q] = wg[q] = 0.0f;
            }
            // Loads' results are first touched one step after the load, and conditions
            // are predicates or address selects, not branches (a divergent branch per
            // element costs more than the work it skips).
            for (int t = -C::PS; t <= steps; ++t) {
                // weights gathered one step ago, for step t + BS - 1
                {
                    const int slot = ((t + C::BS - 1) * C::G + gP) & (C::WS - 1);
#pragma unroll
                    for (int q = 0; q < R; ++q)
                        st_shared((recv >> q) & 1u
                                      ? dump
                                      : wp_base + 4u * (unsigned)(slot * C::MAXK + chain_at<R>(q * 32 + lane)),
                                  wg[q]);
                }
                // step t + BS: the ids and link words loaded one step ago.  Weights that no
                // recent example pushes; where each new weight goes: into its receiver's
                // slot of wp when pushed, else into out (stored through by the write warps)
                recv = ~0u;
                {
                    const int r = (t + C::BS) * C::G + gP;
                    const int xslot = r & (C::XS - 1), wslot = r & (C::WS - 1), oslot = r & (C::OS - 1);
                    if (r >= 0 && r < N) {
                        recv = 0;
#pragma unroll
                        for (int q = 0; q < R; ++q) {
                            const int i = q * 32 + lane, at = chain_at<R>(i);
                            const bool in = i < k, push = in && (lk[q] & LK_PUSH), rc = in && (lk[q] & LK_RECV);
                            wg[q] = ld_if(w + cc[q], in && !rc);
                            recv |= rc ? 1u << q : 0u;
                            const unsigned tslot = ((unsigned)r + ((lk[q] >> 16) & 0xffu)) & (C::WS - 1);
                            const unsigned to =
                                wp_base + 4u * (tslot * C::MAXK + (unsigned)chain_at<R>((int)(lk[q] & 0xffu)));
                            S.pa[xslot][at] = push ? to : in ? out_base + 4u * (unsigned)(oslot * C::MAXK + i) : dump;
                            S.wcol[wslot][i] = in && !push ? cc[q] : -1;
                            S.xa[xslot][at] = in ? xv[q] : -0.0f;
                        }
                        if (lane == 0) S.y[xslot] = yv;
                    }
                }
                // step t + AS: ids, link words, values and label
                {
                    const int r = (t + C::AS) * C::G + gP;
                    k = 0;
                    if (r >= 0 && r < N) {
                        k = (int)(e - b);
                        yv = y[r];
                        const int32_t *cp = col + b + lane;
                        const uint32_t *lp = link + b + lane;
                        const float *vp = val + b + lane;
#pragma unroll
                        for (int q = 0; q < R; ++q)
                            if (q * 32 + lane < k) {
                                cc[q] = __ldcs(cp + q * 32);
                                lk[q] = __ldcs(lp + q * 32);
                                xv[q] = val ? __ldcs(vp + q * 32) : 1.0f;
                            }
                    }
                }
                // row bounds of step t + RS; the rows of step t + PS - 1 into L2 (lane l
                // takes their line l), and the bounds for the next of those
                {
                    const int r = (t + C::RS) * C::G + gP;
                    if (r >= 0 && r < N) {
                        b = row_ptr[r];
                        e = row_ptr[r + 1];
                    }
                    const int64_t pp = pb + 32 * lane;
                    if (lane < R && pp < pe) {
                        prefetch_l2(col + pp);
                        prefetch_l2(link + pp);
                        if (val) prefetch_l2(val + pp);
                    }
                    const int rn = (t + C::PS) * C::G + gP;
                    pb = pe = 0;
                    if (rn >= 0 && rn < N) {
                        pb = row_ptr[rn];
                        pe = row_ptr[rn + 1];
                    }
                }
                __syncthreads();
            }
        }
    } else {
        for (int ep = 0; ep < epochs; ++ep)
            for (int t = -C::PS; t <= steps; ++t) {
                // new weights of step t - 1 that no example among the next D takes on chip go
                // through to global memory (a pushed weight is written again by its
                // receiver, so two stores of one step never hit one address)
                if (gW >= 0 && t >= 1) {
#pragma unroll
                    for (int g = 0; g < C::WPER; ++g) {
                        const int r = (t - 1) * C::G + gW + g;
                        if (r < N) {
                            const int wslot = r & (C::WS - 1), oslot = r & (C::OS - 1);
                            int32_t cj[R];
                            float v[R];
#pragma unroll
                            for (int q = 0; q < R; ++q) {
                                cj[q] = S.wcol[wslot][q * 32 + lane];
                                v[q] = S.out[oslot][q * 32 + lane];
                            }
#pragma unroll
                            for (int q = 0; q < R; ++q)
                                if (cj[q] >= 0) w[cj[q]] = v[q];
                        }
                    }
                }
                __syncthreads();
            }
    }
}

// link[p] (layout above): receive flag from the previous occurrence, push
// target from the next occurrence, each when it lies within D examples
__global__ void k_chain_link(const int32_t *__restrict__ prev, const int32_t *__restrict__ next,
                             const int32_t *__restrict__ row_of, const int64_t *__restrict__ row_ptr, int64_t nnz,
                             uint32_t *__restrict__ link, int D, const int *status)
{
    if (read_status(status)) return;
    for (int64_t p = (int64_t)blockIdx.x * blockDim.x + threadIdx.x; p < nnz; p += (int64_t)gridDim.x * blockDim.x) {
        const int32_t t = row_of[p], q = prev[p], n = next[p];
        uint32_t l = 0;
        if (q >= 0 && t - row_of[q] <= D) l |= LK_RECV;
        if (n >= 0) {
            const int32_t tn = row_of[n];
            if (tn - t <= D) l |= LK_PUSH | ((uint32_t)(tn - t) << 16) | (uint32_t)(n - row_ptr[tn]);
        }
        link[p] = l;
    }
}

}  // namespace

namespace pdb {

int chain_max_row() { return CH_MAXK; }

// registers per lane for the longest example: 1 .. 8 (32 to 256 ids)
static int chain_regs(int64_t max_row) { return max_row <= 32 ? 1 : (int)((max_row + 31) / 32); }

int chain_schedule(const int32_t *prev, const int32_t *next, const int32_t *row_of, const int64_t *row_ptr,
                   int64_t nnz, uint32_t *link, const int *status, cudaStream_t s)
{
    // one forwarding window for every row length
    constexpr int D = ChainCfg<1>::D;
    static_assert(ChainCfg<2>::D == D && ChainCfg<3>::D == D && ChainCfg<4>::D == D && ChainCfg<5>::D == D &&
                  ChainCfg<6>::D == D && ChainCfg<7>::D == D && ChainCfg<8>::D == D, "one window");
    if (nnz > 0) {
        k_chain_link<<<grid_1d(nnz), 256, 0, s>>>(prev, next, row_of, row_ptr, nnz, link, D, status);
        note_launch();
    }
    return cudaPeekAtLastError() == cudaSuccess ? PDB_OK : PDB_ECUDA;
}

using ChainKernel = void (*)(int32_t, const int64_t *, const int32_t *, const float *, const float *,
                             const uint32_t *, float *, float, int, int *, uint64_t *);
struct ChainVariant {
    ChainKernel kern;
    int threads;
    size_t smem;
};

template <int R, bool TRACE>
static ChainVariant chain_variant(int loss)
{
    const ChainKernel kern = loss == PDB_LOSS_LOGISTIC ? k_sgd_chain<R, PDB_LOSS_LOGISTIC, TRACE>
                             : loss == PDB_LOSS_SQUARED ? k_sgd_chain<R, PDB_LOSS_SQUARED, TRACE>
                                                        : k_sgd_chain<R, PDB_LOSS_HINGE, TRACE>;
    return {kern, ChainCfg<R>::THREADS, sizeof(ChainSmem<R>)};
}

template <bool TRACE>
static ChainVariant chain_variant(int R, int loss)
{
    switch (R) {
    case 1: return chain_variant<1, TRACE>(loss);
    case 2: return chain_variant<2, TRACE>(loss);
    case 3: return chain_variant<3, TRACE>(loss);
    case 4: return chain_variant<4, TRACE>(loss);
    case 5: return chain_variant<5, TRACE>(loss);
    case 6: return chain_variant<6, TRACE>(loss);
    case 7: return chain_variant<7, TRACE>(loss);
    default: return chain_variant<8, TRACE>(loss);
    }
}

int chain_run(const pdb_csr *X, const float *y, const uint32_t *link, float *w, int loss, float eta, int epochs,
              int max_row, int *status, uint64_t *trace, cudaStream_t s)
{
    // one kernel per register count (chain_regs), loss (so the gradient has no
    // branch) and whether it stamps an execution trace
    const int R = chain_regs(max_row);
    const ChainVariant v = trace ? chain_variant<true>(R, loss) : chain_variant<false>(R, loss);
    const int variant = ((R - 1) * 3 + (loss >= 0 && loss <= 2 ? loss : 2)) * 2 + (trace ? 1 : 0);
    // set once per device and variant (any device past the table: every call)
    static std::atomic<bool> configured[64][48];
    int dev = 0;
    cudaGetDevice(&dev);
    const bool known = dev >= 0 && dev < 64;
    if (!known || !configured[dev][variant].load(std::memory_order_acquire)) {
        if (cudaFuncSetAttribute((const void *)v.kern, cudaFuncAttributeMaxDynamicSharedMemorySize, (int)v.smem) !=
            cudaSuccess)
            return PDB_ECUDA;
        if (known) configured[dev][variant].store(true, std::memory_order_release);
    }
    v.kern<<<1, v.threads, v.smem, s>>>((int32_t)X->n_rows, X->row_ptr, X->col, X->val, y, link, w, eta, epochs, status,
                                        trace);
    note_launch();
    return cudaPeekAtLastError() == cudaSuccess ? PDB_OK : PDB_ECUDA;
}

}  // namespace pdb
