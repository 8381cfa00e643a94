// Device-side building blocks for sm_103a: PTX wrappers for mbarriers and
// bulk (TMA engine) copies, the P1 element kernels, and block reductions.
#pragma once
#include <cuda_runtime.h>
#include <stdint.h>

#include "layout.h"

namespace ps {

// Bounded waits: an mbarrier wait gives up after this many try_wait rounds
// (each round may itself suspend for a hardware-defined time slice) and a grid
// barrier after this many polls; both then record an error and return.
constexpr uint32_t kMbarSpinLimit = 1u << 22;
constexpr uint32_t kGridSpinLimit = 1u << 26;

enum DevErr : int { kErrNone = 0, kErrMbarTimeout = 1, kErrGridTimeout = 2, kErrBadSize = 4 };

// Per local node, the star passes read the row sum m_l of the chunk's patches
// (layout.h), its sign bit set on Dirichlet nodes (m_l itself is >= 0).
__device__ __forceinline__ bool is_dirichlet(float w) { return __float_as_int(w) < 0; }
__device__ __forceinline__ bool is_dirichlet(double w) { return __double_as_longlong(w) < 0; }

// ---------------------------------------------------------------- PTX: mbarrier + bulk copy
__device__ __forceinline__ uint32_t smem_u32(const void *p) {
    return static_cast<uint32_t>(__cvta_generic_to_shared(p));
}
__device__ __forceinline__ void mbar_init(uint64_t *bar, uint32_t count) {
    asm volatile("mbarrier.init.shared::cta.b64 [%0], %1;" ::"r"(smem_u32(bar)), "r"(count) : "memory");
}
__device__ __forceinline__ void fence_mbar_init() {
    asm volatile("fence.mbarrier_init.release.cluster;" ::: "memory");
}
__device__ __forceinline__ void fence_proxy_async_smem() {
    asm volatile("fence.proxy.async.shared::cta;" ::: "memory");
}
__device__ __forceinline__ void mbar_arrive_expect_tx(uint64_t *bar, uint32_t bytes) {
    asm volatile("mbarrier.arrive.expect_tx.shared::cta.b64 _, [%0], %1;" ::"r"(smem_u32(bar)), "r"(bytes)
                 : "memory");
}
// Global -> shared bulk copy through the TMA engine; completion is signalled
// on `bar` as transaction bytes.  dst, src 16-byte aligned, bytes % 16 == 0.
__device__ __forceinline__ void bulk_g2s(void *dst, const void *src, uint32_t bytes, uint64_t *bar) {
    asm volatile(
        "cp.async.bulk.shared::cluster.global.mbarrier::complete_tx::bytes [%0], [%1], %2, [%3];" ::"r"(
            smem_u32(dst)),
        "l"(src), "r"(bytes), "r"(smem_u32(bar))
        : "memory");
}
// The same for data read once per pass of a working set larger than L2: the
// lines are the first to be replaced, so that they do not push out what the
// next kernels read again.
__device__ __forceinline__ void bulk_g2s_stream(void *dst, const void *src, uint32_t bytes, uint64_t *bar) {
    uint64_t policy;
    asm volatile("createpolicy.fractional.L2::evict_first.b64 %0, 1.0;" : "=l"(policy));
    asm volatile(
        "cp.async.bulk.shared::cluster.global.mbarrier::complete_tx::bytes.L2::cache_hint [%0], [%1], %2, [%3], %4;" ::"r"(
            smem_u32(dst)),
        "l"(src), "r"(bytes), "r"(smem_u32(bar)), "l"(policy)
        : "memory");
}
__device__ __forceinline__ bool mbar_try_wait(uint64_t *bar, uint32_t parity) {
    uint32_t ok;
    asm volatile(
        "{\n\t.reg .pred p;\n\t"
        "mbarrier.try_wait.parity.shared::cta.b64 p, [%1], %2;\n\t"
        "selp.u32 %0, 1, 0, p;\n\t}\n"
        : "=r"(ok)
        : "r"(smem_u32(bar)), "r"(parity)
        : "memory");
    return ok != 0;
}
// Bounded wait for phase `parity` of `bar`.  Returns false on timeout.
__device__ __forceinline__ bool mbar_wait_bounded(uint64_t *bar, uint32_t parity) {
    for (uint32_t i = 0; i < kMbarSpinLimit; ++i)
        if (mbar_try_wait(bar, parity)) return true;
    return false;
}

// ---------------------------------------------------------------- dependent launches
// Between two kernels of one stream, the second launched with
// cudaLaunchAttributeProgrammaticStreamSerialization: once every block of the
// first has passed grid_dep_launch the second's blocks may start, and
// grid_dep_wait holds them until the first has ended and its writes are
// visible.  Without the attribute both do nothing.
__device__ __forceinline__ void grid_dep_launch() { asm volatile("griddepcontrol.launch_dependents;" ::: "memory"); }
__device__ __forceinline__ void grid_dep_wait() { asm volatile("griddepcontrol.wait;" ::: "memory"); }

// ---------------------------------------------------------------- completion counter
// "Last block" detection: every block publishes its partial result with a
// plain store, then increments a device-scope counter with acquire-release
// semantics (no sequentially consistent fence); the block that sees
// count == gridDim - 1 has acquired every other block's partial.
__device__ __forceinline__ unsigned int atomic_add_acq_rel(unsigned int *p, unsigned int v) {
    unsigned int old;
    asm volatile("atom.add.acq_rel.gpu.u32 %0, [%1], %2;" : "=r"(old) : "l"(p), "r"(v) : "memory");
    return old;
}

// ---------------------------------------------------------------- reductions
__device__ __forceinline__ double warp_sum(double v) {
#pragma unroll
    for (int o = 16; o > 0; o >>= 1) v += __shfl_xor_sync(0xffffffffu, v, o);
    return v;
}
// Block-wide sum in a fixed order (the result is bitwise reproducible for a
// given blockDim).  `red` holds >= 32 doubles.  All threads get the result.
__device__ __forceinline__ double block_sum(double v, double *red) {
    const int lane = threadIdx.x & 31, wid = threadIdx.x >> 5, nw = (blockDim.x + 31) >> 5;
    v = warp_sum(v);
    __syncthreads();
    if (lane == 0) red[wid] = v;
    __syncthreads();
    double t = (threadIdx.x < nw) ? red[threadIdx.x] : 0.0;
    if (wid == 0) t = warp_sum(t);
    if (threadIdx.x == 0) red[0] = t;
    __syncthreads();
    double r = red[0];
    __syncthreads();
    return r;
}
// Sum of n doubles in global memory in a fixed order, by one block.
__device__ __forceinline__ double block_sum_array(const double *a, int n, double *red) {
    double s = 0.0;
    for (int i = threadIdx.x; i < n; i += blockDim.x) s += __ldcg(a + i);
    return block_sum(s, red);
}

// ---------------------------------------------------------------- double-float dot accumulation
// FP64 instructions are scarce on this part (2 DFMA/clk/SM), so dot products
// of FP32 vectors are accumulated in "double-float" form: an unevaluated sum
// hi + lo of two floats, updated with Knuth's error-free TwoSum and the
// FMA-based exact product (Dekker / Ogita-Rump-Oishi "Dot2").  The result is
// as accurate as a sum carried in twice the FP32 precision; it is converted to
// FP64 once per warp and the per-warp values are summed in FP64 in a fixed
// order.  The intrinsics below are never contracted or reassociated.
struct DotF {
    float hi = 0.f, lo = 0.f;
    __device__ __forceinline__ void add(float v) {
        const float s = __fadd_rn(hi, v);
        const float bb = __fsub_rn(s, hi);
        const float e = __fadd_rn(__fsub_rn(hi, __fsub_rn(s, bb)), __fsub_rn(v, bb));
        hi = s;
        lo = __fadd_rn(lo, e);
    }
    __device__ __forceinline__ void add_prod(float a, float b) {
        const float p = __fmul_rn(a, b);
        const float pe = __fmaf_rn(a, b, -p);
        const float s = __fadd_rn(hi, p);
        const float bb = __fsub_rn(s, hi);
        const float e = __fadd_rn(__fsub_rn(hi, __fsub_rn(s, bb)), __fsub_rn(p, bb));
        hi = s;
        lo = __fadd_rn(lo, __fadd_rn(e, pe));
    }
    __device__ __forceinline__ void merge(float h2, float l2) {
        const float s = __fadd_rn(hi, h2);
        const float bb = __fsub_rn(s, hi);
        const float e = __fadd_rn(__fsub_rn(hi, __fsub_rn(s, bb)), __fsub_rn(h2, bb));
        hi = s;
        lo = __fadd_rn(__fadd_rn(lo, l2), e);
    }
};
// FP64 accumulator with the same interface (FP64 vectors).
struct DotD {
    double v = 0.0;
    __device__ __forceinline__ void add(double x) { v += x; }
    __device__ __forceinline__ void add_prod(double a, double b) { v = fma(a, b, v); }
};
template <typename T> struct DotOf;
template <> struct DotOf<float> { using type = DotF; };
template <> struct DotOf<double> { using type = DotD; };

// Block-wide sum of accumulators in a fixed order; all threads get the FP64
// result.  `red` holds >= 32 doubles.
__device__ __forceinline__ double block_sum(const DotF &a, double *red) {
    float hi = a.hi, lo = a.lo;
#pragma unroll
    for (int o = 16; o > 0; o >>= 1) {
        const float h2 = __shfl_xor_sync(0xffffffffu, hi, o);
        const float l2 = __shfl_xor_sync(0xffffffffu, lo, o);
        DotF t;
        t.hi = hi;
        t.lo = lo;
        t.merge(h2, l2);
        hi = t.hi;
        lo = t.lo;
    }
    const int lane = threadIdx.x & 31, wid = threadIdx.x >> 5, nw = (blockDim.x + 31) >> 5;
    __syncthreads();
    if (lane == 0) red[wid] = (double)hi + (double)lo;
    __syncthreads();
    if (threadIdx.x == 0) {
        double t = 0.0;
        for (int w = 0; w < nw; ++w) t += red[w];
        red[32] = t;
    }
    __syncthreads();
    const double r = red[32];
    __syncthreads();
    return r;
}
__device__ __forceinline__ double block_sum(const DotD &a, double *red) { return block_sum(a.v, red); }

// N block sums (N <= 3) with one set of barriers; each result is bitwise the
// one block_sum gives (same per-warp values, same fixed-order sums).  Blocks
// of at most 256 threads; `red` holds >= 34 doubles.
__device__ __forceinline__ float2 warp_dotf(const DotF &a) {
    float hi = a.hi, lo = a.lo;
#pragma unroll
    for (int o = 16; o > 0; o >>= 1) {
        const float h2 = __shfl_xor_sync(0xffffffffu, hi, o);
        const float l2 = __shfl_xor_sync(0xffffffffu, lo, o);
        DotF t;
        t.hi = hi;
        t.lo = lo;
        t.merge(h2, l2);
        hi = t.hi;
        lo = t.lo;
    }
    return make_float2(hi, lo);
}
template <int N>
__device__ __forceinline__ void block_sum_n(const DotF *a, double *red, double *out) {
    float2 w[N];
#pragma unroll
    for (int k = 0; k < N; ++k) w[k] = warp_dotf(a[k]);
    const int lane = threadIdx.x & 31, wid = threadIdx.x >> 5, nw = (blockDim.x + 31) >> 5;
    __syncthreads();
    if (lane == 0) {
#pragma unroll
        for (int k = 0; k < N; ++k) red[8 * k + wid] = (double)w[k].x + (double)w[k].y;
    }
    __syncthreads();
    if (lane == 0 && wid < N) {
        double t = 0.0;
        for (int v = 0; v < nw; ++v) t += red[8 * wid + v];
        red[24 + wid] = t;
    }
    __syncthreads();
#pragma unroll
    for (int k = 0; k < N; ++k) out[k] = red[24 + k];
    __syncthreads();
}
__device__ __forceinline__ void block_sum2(const DotF &a, const DotF &b, double *red, double &ra, double &rb) {
    const DotF v[2] = {a, b};
    double o[2];
    block_sum_n<2>(v, red, o);
    ra = o[0];
    rb = o[1];
}

// ---------------------------------------------------------------- P1 star patches
// One thread evaluates a whole star patch (layout.h) from its weights:
//   out_i = sum over the patch's edges (i, j) of A^s_ij (v_j - v_i).
// The row-sum term m_i v_i is added once per local node (mrow).  Per edge
// one difference and two multiply-adds: 57 operations for the 19 edges of a
// closed star of six tetrahedra, against ~55 for each of its tetrahedra when
// the element matrices are applied one by one.
// out[slot]: 0 -> a, 1 -> b (3D), 2 + j -> r_j, j < nr; other slots untouched.
struct StarIds {
    uint32_t w[kStarIds];
    __device__ __forceinline__ int nr() const { return (int)((w[4] >> 16) & 7u); }
    __device__ __forceinline__ bool closed() const { return (w[4] >> 20) & 1u; }
    // byte offsets of an FP32 value per node
    __device__ __forceinline__ uint32_t a() const { return w[0] & 0xffffu; }
    __device__ __forceinline__ uint32_t b() const { return w[0] >> 16; }
    __device__ __forceinline__ uint32_t ring(int j) const {
        return j & 1 ? w[1 + j / 2] >> 16 : w[1 + j / 2] & 0xffffu;
    }
};
// A node's value from its byte offset of an FP32 value.
template <typename T>
__device__ __forceinline__ T node_value(const T *__restrict__ s_val, uint32_t off) {
    return *reinterpret_cast<const T *>(reinterpret_cast<const char *>(s_val) + off * (sizeof(T) / 4));
}

// FP32: the whole record in registers.  rec: the patch's entry of row 0.  The
// rows of a star of up to six ring nodes are loaded before its size is known.
template <int D>
struct StarF {
    uint4 v[kStarVec<D>];
    __device__ __forceinline__ uint32_t word(int k) const {
        const uint4 &q = v[k / 4];
        return k % 4 == 0 ? q.x : k % 4 == 1 ? q.y : k % 4 == 2 ? q.z : q.w;
    }
    __device__ __forceinline__ float weight(int k) const { return __uint_as_float(word(kStarIds + k)); }
    __device__ __forceinline__ StarIds ids() const {
        return StarIds{{word(0), word(1), word(2), word(3), word(4)}};
    }
    __device__ __forceinline__ void load(const uint4 *__restrict__ rec) {
        constexpr int n = D == 3 ? 6 : kStarVec<D>;
#pragma unroll
        for (int k = 0; k < n; ++k) v[k] = __ldg(rec + k * kStarLanes);
        if (D == 3 && ids().nr() == 7) v[6] = __ldg(rec + 6 * kStarLanes);
    }
    __device__ __forceinline__ void load_shared(const uint4 *rec) {
        constexpr int n = D == 3 ? 6 : kStarVec<D>;
#pragma unroll
        for (int k = 0; k < n; ++k) v[k] = rec[k * kStarLanes];
        if (D == 3 && ids().nr() == 7) v[6] = rec[6 * kStarLanes];
    }
};
// FP64 weights of a star of NR ring nodes.
template <int D, int NR>
struct StarD {
    static constexpr int n = D == 3 ? (4 + 3 * (NR - 1) + 1) / 2 : (2 + 2 * (NR - 1)) / 2;
    double2 v[n];
    __device__ __forceinline__ double weight(int k) const { return k & 1 ? v[k / 2].y : v[k / 2].x; }
    __device__ __forceinline__ void load(const double2 *__restrict__ wt) {
#pragma unroll
        for (int k = 0; k < n; ++k) v[k] = __ldg(wt + k * kStarLanes);
    }
};

template <int D, int NR, typename T, typename W>
__device__ __forceinline__ void star_eval_nr(const W &S, const StarIds &id, const T *__restrict__ s_val,
                                             T *__restrict__ out) {
    constexpr int w0 = D == 3 ? 2 : 1;   // first weight of ring node 0
    const T va = node_value(s_val, id.a());
    T vb = T(0), oa = T(0), ob = T(0);
    if (D == 3) {
        vb = node_value(s_val, id.b());
        oa = S.weight(0) * (vb - va);
        ob = -oa;
    }
    T v0 = T(0), first = T(0), pv = T(0), po = T(0);
#pragma unroll
    for (int j = 0; j < NR; ++j) {
        const int w = j == 0 ? w0 : w0 + (D - 1) + D * (j - 1);
        const T v = node_value(s_val, id.ring(j));
        T d = v - va;
        oa = fma(S.weight(w), d, oa);
        T o = -(S.weight(w) * d);
        if (D == 3) {
            d = v - vb;
            ob = fma(S.weight(w + 1), d, ob);
            o = fma(-S.weight(w + 1), d, o);
        }
        if (j == 0) {
            v0 = v;
        } else {
            d = v - pv;
            po = fma(S.weight(w + D - 1), d, po);
            o = fma(-S.weight(w + D - 1), d, o);
            if (j == 1) first = po; else out[2 + j - 1] = po;
        }
        pv = v;
        po = o;
    }
    const T wrap = S.weight(D == 3 ? 1 : 0);
    // (an open star's weight is 0, but its ends are no neighbours: an infinite
    // value at one leaves the other's row alone)
    const T d = id.closed() ? v0 - pv : T(0);
    out[2 + NR - 1] = fma(wrap, d, po);
    out[2] = fma(-wrap, d, first);
    out[0] = oa;
    if (D == 3) out[1] = ob;
}
template <int D>
__device__ __forceinline__ void star_eval(const StarF<D> &S, const float *__restrict__ s_val, float *__restrict__ out) {
    const StarIds id = S.ids();
    switch (id.nr()) {
        case 6: star_eval_nr<D, 6>(S, id, s_val, out); break;
        case 7: star_eval_nr<D, 7>(S, id, s_val, out); break;
        case 5: star_eval_nr<D, 5>(S, id, s_val, out); break;
        case 4: star_eval_nr<D, 4>(S, id, s_val, out); break;
        case 3: star_eval_nr<D, 3>(S, id, s_val, out); break;
        default: star_eval_nr<D, 2>(S, id, s_val, out); break;
    }
}
// One code path for every star but the closed one of six: seven ring nodes,
// the ones past nr with zero weights (whatever node their id names) and
// contributions nobody reads; the edge (r_{nr-1}, r_0) is added at the end.
// For kernels that run all their phases in a loop, where the instruction
// cache pays for every variant, and for warps of stars of many sizes.  STRICT:
// a node past nr that is infinite or NaN adds nothing either.
template <int D, bool STRICT = false, typename T, typename W>
__device__ __forceinline__ void star_eval_any(const W &S, const StarIds &id, const T *__restrict__ s_val,
                                              T *__restrict__ out) {
    constexpr int w0 = D == 3 ? 2 : 1;
    const int nr = id.nr();
    const T va = node_value(s_val, id.a());
    T vb = T(0), oa = T(0), ob = T(0);
    if (D == 3) {
        vb = node_value(s_val, id.b());
        oa = S.weight(0) * (vb - va);
        ob = -oa;
    }
    T pv = T(0), po = T(0);
#pragma unroll
    for (int j = 0; j < kStarRing; ++j) {
        const int w = j == 0 ? w0 : w0 + (D - 1) + D * (j - 1);
        const bool none = STRICT && j >= 2 && j >= nr;
        const T v = node_value(s_val, id.ring(j));
        T d = none ? T(0) : v - va;
        oa = fma(S.weight(w), d, oa);
        T o = -(S.weight(w) * d);
        if (D == 3) {
            d = none ? T(0) : v - vb;
            ob = fma(S.weight(w + 1), d, ob);
            o = fma(-S.weight(w + 1), d, o);
        }
        if (j > 0) {
            d = none ? T(0) : v - pv;
            out[2 + j - 1] = fma(S.weight(w + D - 1), d, po);
            o = fma(-S.weight(w + D - 1), d, o);
        }
        pv = v;
        po = o;
    }
    out[2 + kStarRing - 1] = po;
    out[0] = oa;
    if (D == 3) out[1] = ob;
    const T wrap = S.weight(D == 3 ? 1 : 0);
    if (wrap != T(0)) {
        const int last = nr - 1;
        uint32_t w = id.w[1];
        if (last >= 2) w = id.w[2];
        if (last >= 4) w = id.w[3];
        if (last >= 6) w = id.w[4];
        const uint32_t off = last & 1 ? w >> 16 : w & 0xffffu;
        const T f = wrap * (node_value(s_val, id.ring(0)) - node_value(s_val, off));
        out[2 + last] += f;
        out[2] -= f;
    }
}
__device__ __forceinline__ StarIds star_ids(const uint4 *__restrict__ rec) {
    const uint4 q = __ldg(rec);
    return StarIds{{q.x, q.y, q.z, q.w, __ldg(reinterpret_cast<const uint32_t *>(rec + kStarLanes))}};
}
template <int D, int NR>
__device__ __forceinline__ void star_eval64_nr(const double2 *__restrict__ wt, const StarIds &id,
                                               const double *__restrict__ s_val, double *__restrict__ out) {
    StarD<D, NR> S;
    S.load(wt);
    star_eval_nr<D, NR>(S, id, s_val, out);
}
template <int D>
__device__ __forceinline__ void star_eval64(const StarIds &id, const double2 *__restrict__ wt,
                                            const double *__restrict__ s_val, double *__restrict__ out) {
    if (D == 2) {
        // A 2D chunk has stars of every size in one warp: a variant and its
        // loads per size ran one after another (64 x 64 squares, apply in a
        // graph: 10.6 us per size, 8.3 as six and others, 7.4 as one).
        StarD<D, kStarRing> S;
        S.load(wt);
        star_eval_any<D, true>(S, id, s_val, out);
        return;
    }
    switch (id.nr()) {
        case 6: star_eval64_nr<D, 6>(wt, id, s_val, out); break;
        case 7: star_eval64_nr<D, 7>(wt, id, s_val, out); break;
        case 5: star_eval64_nr<D, 5>(wt, id, s_val, out); break;
        case 4: star_eval64_nr<D, 4>(wt, id, s_val, out); break;
        case 3: star_eval64_nr<D, 3>(wt, id, s_val, out); break;
        default: star_eval64_nr<D, 2>(wt, id, s_val, out); break;
    }
}

// Weights and row sums of one patch from its elements: with cm = |T| d! /
// (d+3)! (= |det|/720 in 3D, |det|/120 in 2D) and S the sum of an element's
// alpha (int lambda^a = d! |T| prod(a_i!) / (d + sum a_i)!),
//   consistent: A_ij = b G_ij + cm (S + alpha_i + alpha_j),  m_i = (d+3) cm (S + alpha_i)
//   lumped:     A_ij = b G_ij,                               m_i = |det|/(d+1)! alpha_i
// with b = beta dt^2 and G_ij = c_i . c_j / (d! |det|) the element's stiffness
// weights, computed once per mesh (kGeoWords).  geo: the patch's entry of row
// 0 of element 0; bd: its elements' beta dt^2; al: alpha of the local nodes;
// w32, w64: the patch's record and weights; mass[slot]: the row sums.
template <int D>
__device__ __forceinline__ void star_build(const StarIds &id, const double *__restrict__ geo,
                                           const double (&bd)[kPatchMax], const double *__restrict__ al, bool lumped,
                                           float *__restrict__ w32, double *__restrict__ w64,
                                           double *__restrict__ mass) {
    constexpr int GW = kGeoWords<D>;
    const int nr = id.nr();
    const bool closed = id.closed();
    const int m = closed ? nr : nr - 1;
    auto alpha_of = [&](uint32_t off) { return fabs(node_value(al, off)); };
    const double aa = alpha_of(id.a()), ab = D == 3 ? alpha_of(id.b()) : 0.0;
    const double cmf = lumped ? 0.0 : (D == 3 ? 1.0 / 720.0 : 1.0 / 120.0);
    const double clf = D == 3 ? 1.0 / 24.0 : 1.0 / 6.0;
    double wab = 0.0, ma = 0.0, mb = 0.0;
    double wa0 = 0.0, wb0 = 0.0, m0 = 0.0;           // ring node 0 (a closed star's last element adds to it)
    double pa = 0.0, pb = 0.0, pm = 0.0, wrap = 0.0; // the current ring node, its edge to the next element's
    auto put = [&](int k, double v) {                // weight k
        w64[(k / 2) * 2 * kStarLanes + k % 2] = v;
        w32[((kStarIds + k) / 4) * 4 * kStarLanes + (kStarIds + k) % 4] = (float)v;
    };
    auto first_w = [](int j) { return (D == 3 ? 4 : 2) + D * (j - 1); };   // first weight of ring node j >= 1
    double a0 = alpha_of(id.ring(0));
    // the next element's words are loaded while this one is computed
    double gc[GW], gn[GW];
#pragma unroll
    for (int k = 0; k < GW; ++k) gn[k] = __ldg(geo + k * kStarLanes);
#pragma unroll
    for (int j = 0; j < kPatchMax; ++j) {
        if (j >= m) break;
#pragma unroll
        for (int k = 0; k < GW; ++k) gc[k] = gn[k];
        if (j + 1 < kPatchMax && j + 1 < m) {
#pragma unroll
            for (int k = 0; k < GW; ++k) gn[k] = __ldg(geo + ((j + 1) * GW + k) * kStarLanes);
        }
        const bool last = closed && j == m - 1;
        const double a1 = alpha_of(last ? id.ring(0) : id.ring(j + 1));
        const double b = bd[j];
        const double gAB = D == 3 ? gc[0] : 0.0, gA0 = gc[D == 3 ? 1 : 0], gA1 = gc[D == 3 ? 2 : 1];
        const double gB0 = D == 3 ? gc[3] : 0.0, gB1 = D == 3 ? gc[4] : 0.0, g01 = gc[D == 3 ? 5 : 2];
        const double ad = gc[GW - 1];
        const double cm = ad * cmf;
        const double S = (aa + ab) + (a0 + a1);
        const double sa = S + aa, sb = S + ab, s0 = S + a0, s1 = S + a1;
        if (lumped) {
            const double cl = ad * clf;
            ma = fma(cl, aa, ma);
            mb = fma(cl, ab, mb);
            pm = fma(cl, a0, pm);
        } else {
            const double cr = (D + 3) * cm;
            ma = fma(cr, sa, ma);
            mb = fma(cr, sb, mb);
            pm = fma(cr, s0, pm);
        }
        if (D == 3) {
            wab = fma(b, gAB, fma(cm, sa + ab, wab));
            pb = fma(b, gB0, fma(cm, sb + a0, pb));
        }
        pa = fma(b, gA0, fma(cm, sa + a0, pa));
        const double w01 = fma(b, g01, cm * (s0 + a1));
        // ring node j is complete, except node 0 (the wrapping element may add to it)
        if (j == 0) {
            wa0 = pa;
            wb0 = pb;
            m0 = pm;
        } else {
            put(first_w(j), pa);
            if (D == 3) put(first_w(j) + 1, pb);
            mass[2 + j] = pm;
        }
        pa = fma(b, gA1, cm * (sa + a1));
        pb = D == 3 ? fma(b, gB1, cm * (sb + a1)) : 0.0;
        pm = lumped ? ad * clf * a1 : (D + 3) * cm * s1;
        if (last) {
            wa0 += pa;
            wb0 += pb;
            m0 += pm;
            wrap = w01;
        } else {
            // edge (r_j, r_{j+1}) belongs to ring node j + 1
            put(first_w(j + 1) + D - 1, w01);
        }
        a0 = a1;
    }
    if (!closed) {
        put(first_w(m), pa);
        if (D == 3) put(first_w(m) + 1, pb);
        mass[2 + m] = pm;
    }
    if (D == 3) {
        put(0, wab);
        put(1, wrap);
        put(2, wa0);
        put(3, wb0);
        mass[1] = mb;
    } else {
        put(0, wrap);
        put(1, wa0);
    }
    mass[2] = m0;
    mass[0] = ma;
}

}  // namespace ps
