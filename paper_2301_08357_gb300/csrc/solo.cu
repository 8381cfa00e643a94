// On-chip CG of one mesh: see solo.h.
//
// A mesh of up to a few hundred thousand nodes spends a CG iteration of
// separate kernels waiting: for launches, for chains of dependent loads (chunk
// descriptor, ids, vectors, partial sums) and for grid reductions.  Here one
// cooperative kernel runs the whole inner solve.  Each block owns a contiguous
// range of star patches and keeps in shared memory, for the unknowns they
// touch, every CG vector, the incidence lists and the contributions, and in
// registers the first stars' weights; per iteration it exchanges only
//   * the partial sums of the unknowns it shares with other blocks, and
//   * its shares of the three dot products,
// through L2.  The recurrences are the one-reduction form of cg1.cuh
// (Chronopoulos and Gear), so there is one exchange per iteration: a block
// stores its shares into every block's own list, each block waits for its
// list, sums it in a fixed order and advances the scalars (the same words in
// the same order, so all take the same decision); the others' partial sums
// travel, and are read, at the same time.  Every word exchanged carries the iteration's tag
// beside 32 bits of its value, so a reader knows a word by itself: no fence,
// no barrier counter, no clearing between iterations.  Two buffers suffice: a
// block overwrites a word of iteration k in iteration k + 2, after it has seen
// every block's share of k + 1, which that block stored after its last read of
// iteration k.  One list per reader costs n^2 words, but a list that all
// blocks poll took 4 us to arrive (150 readers of the same lines), and a
// reducing block in between two hops of 1.7 us.
// Results are bitwise reproducible (fixed orders).  Every wait is bounded; on
// expiry the error flag is set and the kernel ends.
#include <cuda_runtime.h>

#include <algorithm>
#include <cmath>
#include <cstring>

#include "../../include/pressure.h"
#include "internal.h"
#include "batched.h"
#include "cg1.cuh"

namespace ps {

// ---------------------------------------------------------------- host layout
constexpr int kSoloResident = 2;   // stars per thread whose FP32 record stays in registers
static SoloSmem solo_smem(const SoloPrep &p, int esz) {
    SoloSmem L;
    uint64_t off = 0;
    auto take = [&](uint64_t bytes) {
        const uint64_t at = off;
        off += (bytes + 15) / 16 * 16;
        return (uint32_t)at;
    };
    const uint64_t v = (uint64_t)p.max_loc * esz;
    L.val = take(v);
    L.r = take(v);
    L.s = take(v);
    L.p = take(v);
    L.x = take(v);
    L.di = take(v);
    L.m = take(v);
    L.w = take(v);
    L.contrib = take(((uint64_t)p.max_star * kPatchSlots + 1) * esz);
    L.goff = take(((uint64_t)p.max_loc / 32 + 2) * 4);
    L.ell = take((uint64_t)p.max_ell * 4);
    L.sh = take((uint64_t)p.max_sh * 16);
    L.total = (uint32_t)std::min<uint64_t>(off, UINT32_MAX);
    return L;
}

// ---------------------------------------------------------------- kernel
template <typename T>
struct SoloArgs {
    const SoloBlock *blocks;
    const uint4 *ids4;
    const uint32_t *ids1;
    const int32_t *gid;
    const uint32_t *goff, *ell;
    const int4 *sh;
    const uint4 *srec;
    int srows;
    const double2 *sw64;
    const T *dinv, *mtot;
    uint2 *part0, *part1;       // [n_slots * kWords] partial sums, two buffers
    int n_slots;
    const double *r64;
    double *x64;
    double scale, inv_scale, tol2;
    int relative, nan_breaks;
    int drop;                   // 1: a breakdown leaves x64 alone, 0: it keeps the last iterate
    uint32_t spin_limit;        // polls of a wait before it gives up
    uint32_t nap;               // ns before an iteration's first poll (solo_nap)
    uint32_t *beat;             // in a batch: counts its runs' iterations by 256 and their ends (null: a run alone)
    long long max_iters;
    uint4 *exch;                // [2 buffers][reader][3 products][writer], two tagged words each
    uint32_t tag0;              // tag of the first iteration
    CgState *st;
    int *err;
    SoloSmem L;
};

// What blocks exchange travels in 8-byte words {32 bits of the value, tag}: a
// word is read and written as a whole, and it is valid when its tag is the
// iteration's.  No word has to be ordered against another, so neither side
// needs a fence.
__device__ __forceinline__ void st_tagged(uint2 *p, uint32_t v, uint32_t tag) {
    const unsigned long long w = (unsigned long long)v | (unsigned long long)tag << 32;
    asm volatile("st.relaxed.gpu.global.u64 [%0], %1;" ::"l"(p), "l"(w) : "memory");
}
__device__ __forceinline__ uint2 ld_tagged(const uint2 *p) {
    unsigned long long w;
    asm volatile("ld.relaxed.gpu.global.u64 %0, [%1];" : "=l"(w) : "l"(p) : "memory");
    return make_uint2((uint32_t)w, (uint32_t)(w >> 32));
}
// Two words at once (each valid by its own tag).
__device__ __forceinline__ void st_pair(uint4 *p, uint32_t v0, uint32_t v1, uint32_t tag) {
    const unsigned long long t = (unsigned long long)tag << 32;
    asm volatile("st.relaxed.gpu.global.v2.u64 [%0], {%1, %2};" ::"l"(p), "l"(t | v0), "l"(t | v1) : "memory");
}
__device__ __forceinline__ uint4 ld_pair(const uint4 *p) {
    unsigned long long a, b;
    asm volatile("ld.relaxed.gpu.global.v2.u64 {%0, %1}, [%2];" : "=l"(a), "=l"(b) : "l"(p) : "memory");
    return make_uint4((uint32_t)a, (uint32_t)(a >> 32), (uint32_t)b, (uint32_t)(b >> 32));
}
__device__ __forceinline__ uint32_t ld_relaxed(const uint32_t *p) {
    uint32_t v;
    asm volatile("ld.relaxed.gpu.global.u32 %0, [%1];" : "=r"(v) : "l"(p) : "memory");
    return v;
}
// The first wait of a run in a batch lasts until thread blocks that still run
// earlier meshes come to this one, which may be many runs: past the first polls
// it is waited for here.  The polls are counted from the last sign of life of any
// run (the beat), and the wait ends at once when some other wait has given up.
__device__ __noinline__ bool solo_queue_wait(const uint2 *word, uint32_t tag, const uint32_t *beat, const int *err) {
    uint32_t seen = ld_relaxed(beat);
    for (uint32_t polls = 0; polls < kGridSpinLimit; ++polls) {
        if (ld_tagged(word).y == tag) return true;
        if (ld_relaxed(reinterpret_cast<const uint32_t *>(err))) return false;
        const uint32_t now = ld_relaxed(beat);
        if (now != seen) polls = 0;
        seen = now;
        __nanosleep(64);
    }
    return false;
}
// A wait's budget: false once it has given up.  The polls are set to 0 before
// every wait (a budget spent over a whole run ended healthy long runs, and after
// its first 4,096 polls every later one slept).
struct Spin {
    uint32_t polls = 0;
    bool ok = true;
    __device__ __forceinline__ bool again(uint32_t limit) {
        if (++polls >= limit) ok = false;
        if (polls > 4096u) __nanosleep(64);
        return ok;
    }
    // in the first wait of a run in a batch
    __device__ __forceinline__ bool again_queued(const uint2 *word, uint32_t tag, const uint32_t *beat, const int *err) {
        if (++polls >= 1024u) ok = solo_queue_wait(word, tag, beat, err);
        return ok;
    }
};
// A value of type T in kWords words per entry; word k of entry e of n at
// [k * n + e].
template <typename T> struct Tagged;
template <> struct Tagged<float> {
    static constexpr int kWords = 1;
    static __device__ __forceinline__ void put(uint2 *p, int, int e, float v, uint32_t tag) {
        st_tagged(p + e, __float_as_uint(v), tag);
    }
    static __device__ __forceinline__ float of(const uint2 *w) { return __uint_as_float(w[0].x); }
};
template <> struct Tagged<double> {
    static constexpr int kWords = 2;
    static __device__ __forceinline__ void put(uint2 *p, int n, int e, double v, uint32_t tag) {
        const unsigned long long b = (unsigned long long)__double_as_longlong(v);
        st_tagged(p + e, (uint32_t)b, tag);
        st_tagged(p + n + e, (uint32_t)(b >> 32), tag);
    }
    static __device__ __forceinline__ double of(const uint2 *w) { return __hiloint2double((int)w[1].x, (int)w[0].x); }
};

// A dot product's share: a float pair (unevaluated sum) for FP32 vectors, a
// double for FP64 ones; two words either way.  Inside a warp pairs are added as
// pairs; above it, where the rounding of a single addition still shows in the
// total, as three floats (Wide), which lose nothing that a double would keep.
// FP64 additions there were slower (a warp's takes its SM sub-partition 64
// cycles: 301 x 301 squares 10% per solve).  Relative error of a total against
// exact sums, rms over random vectors of 4,225 to 274,625 nodes: pairs
// throughout 1.6e-15 to 2.4e-15, the fused pass of cg1.cuh 5.1e-16 to 8.0e-16,
// this 3.2e-16 to 4.3e-16.
template <typename T> struct Share;
template <> struct Share<float> {
    using type = float2;
    struct Wide {
        float hi, lo, t;
    };
    static __device__ __forceinline__ float2 zero() { return make_float2(0.f, 0.f); }
    static __device__ __forceinline__ float2 add(float2 a, float2 b) {
        DotF t;
        t.hi = a.x;
        t.lo = a.y;
        t.merge(b.x, b.y);
        return make_float2(t.hi, t.lo);
    }
    static __device__ __forceinline__ float2 of(const DotF &a) { return make_float2(a.hi, a.lo); }
    static __device__ __forceinline__ float2 shfl(float2 a, int o) {
        return make_float2(__shfl_xor_sync(0xffffffffu, a.x, o), __shfl_xor_sync(0xffffffffu, a.y, o));
    }
    static __device__ __forceinline__ float2 from(uint32_t x, uint32_t y) {
        return make_float2(__uint_as_float(x), __uint_as_float(y));
    }
    static __device__ __forceinline__ Wide wide(float2 a) { return {a.x, a.y, 0.f}; }
    // s + e = a + b exactly (Knuth's TwoSum)
    static __device__ __forceinline__ float two_sum(float a, float b, float &e) {
        const float s = __fadd_rn(a, b), bb = __fsub_rn(s, a);
        e = __fadd_rn(__fsub_rn(a, __fsub_rn(s, bb)), __fsub_rn(b, bb));
        return s;
    }
    static __device__ __forceinline__ Wide add(Wide a, Wide b) {
        float e, f, g;
        Wide o;
        o.hi = two_sum(a.hi, b.hi, e);
        const float u = two_sum(a.lo, b.lo, f);
        o.lo = two_sum(u, e, g);
        o.t = __fadd_rn(__fadd_rn(a.t, b.t), __fadd_rn(f, g));
        return o;
    }
    static __device__ __forceinline__ Wide shfl(Wide a, int o) {
        return {__shfl_xor_sync(0xffffffffu, a.hi, o), __shfl_xor_sync(0xffffffffu, a.lo, o),
                __shfl_xor_sync(0xffffffffu, a.t, o)};
    }
    static __device__ __forceinline__ uint2 bits(Wide a) {
        // hi + lo renormalised (|lo| is far below |hi|), then t into the rest
        const float s = __fadd_rn(a.hi, a.lo), r = __fsub_rn(a.lo, __fsub_rn(s, a.hi));
        return make_uint2(__float_as_uint(s), __float_as_uint(__fadd_rn(r, a.t)));
    }
    static __device__ __forceinline__ double total(Wide a) { return (double)a.hi + ((double)a.lo + (double)a.t); }
};
template <> struct Share<double> {
    using type = double;
    using Wide = double;
    static __device__ __forceinline__ double zero() { return 0.0; }
    static __device__ __forceinline__ double add(double a, double b) { return a + b; }
    static __device__ __forceinline__ double of(const DotD &a) { return a.v; }
    static __device__ __forceinline__ double shfl(double a, int o) { return __shfl_xor_sync(0xffffffffu, a, o); }
    static __device__ __forceinline__ double wide(double a) { return a; }
    static __device__ __forceinline__ uint2 bits(double a) {
        return make_uint2((uint32_t)__double2loint(a), (uint32_t)__double2hiint(a));
    }
    static __device__ __forceinline__ double from(uint32_t x, uint32_t y) { return __hiloint2double((int)y, (int)x); }
    static __device__ __forceinline__ double total(double a) { return a; }
};
// Sum of each group of N lanes, in all of them.
template <typename T, int N>
__device__ __forceinline__ typename Share<T>::Wide sum_lanes(typename Share<T>::Wide v) {
#pragma unroll
    for (int o = N / 2; o > 0; o >>= 1) v = Share<T>::add(v, Share<T>::shfl(v, o));
    return v;
}
// Three warp sums at once: after two exchanges each lane carries one product
// (lane / 8 = 0: a, 1: b, 2: c), which three more add up -- six additions per
// lane instead of fifteen.  Lanes 0, 8 and 16 hold the results.
template <typename T>
__device__ __forceinline__ typename Share<T>::type warp_share3(typename Share<T>::type a, typename Share<T>::type b,
                                                               typename Share<T>::type c, int lane) {
    using Sh = Share<T>;
    const bool up = lane & 16;
    // lanes of the lower half keep a and b, those of the upper half c
    typename Sh::type k0 = Sh::add(up ? c : a, Sh::shfl(up ? a : c, 16));
    typename Sh::type k1 = Sh::add(up ? Sh::zero() : b, Sh::shfl(up ? b : Sh::zero(), 16));
    const bool odd = lane & 8;
    typename Sh::type v = Sh::add(odd ? k1 : k0, Sh::shfl(odd ? k0 : k1, 8));
#pragma unroll
    for (int o = 4; o > 0; o >>= 1) v = Sh::add(v, Sh::shfl(v, o));
    return v;
}
__device__ __forceinline__ bool finite(double v) { return (__double2hiint(v) & 0x7fffffff) < 0x7ff00000; }
// Positive (not 0, not NaN), from the sign and exponent word.
__device__ __forceinline__ bool positive(double v) {
    const int h = __double2hiint(v);
    return h > 0 && h <= 0x7ff00000;
}

template <typename T>
__device__ __forceinline__ T fma_rn(T a, T b, T c);
template <>
__device__ __forceinline__ float fma_rn(float a, float b, float c) { return __fmaf_rn(a, b, c); }
template <>
__device__ __forceinline__ double fma_rn(double a, double b, double c) { return __fma_rn(a, b, c); }

// The scalars of a run, advanced once per iteration by one warp of every
// block from the same totals.
template <typename T>
struct SoloScalars {
    double rz = 0.0, ra = 0.0, rr0 = 0.0, stop_rr = 0.0;   // gamma; gamma * alpha
    long long iters = 0;
    int status = kCgRunning;
    // g, d, rho: gamma, delta, rho of iteration `it` in every lane.  quot: alpha in
    // lane 0, beta in lane 1.  Returns 1 if the run ends.
    __device__ __forceinline__ int advance(const SoloArgs<T> &A, int bid, int it, double g, double d, double rho, int lane,
                                           double &quot) {
        int done = 0;
        // alpha' = g / (d - beta g / alpha) = g (rz alpha) / (d (rz alpha) - g g), beta = g / rz
        const double num = it == 0 || lane == 1 ? g : g * ra;
        const double den = it == 0 ? d : lane == 1 ? rz : d * ra - g * g;
        quot = num / den;
        if (it == 0) {
            rr0 = rho;
            stop_rr = A.relative ? A.tol2 * rho : A.tol2;
            if (A.nan_breaks && !finite(rho)) {
                done = 1;
                status = kCgBreakdown;
            } else if (!(rho > 0.0) || (!A.relative && rho <= stop_rr)) {
                done = 1;
                status = kCgConverged;
            } else if (!positive(d) || !finite(g) || !finite(d)) {
                done = 1;
                status = kCgBreakdown;
            }
        } else {
            iters += 1;
            const bool pos = __shfl_sync(0xffffffffu, positive(den) ? 1 : 0, 0) && positive(ra);
            const bool fin = finite(g) && finite(d) && finite(rho);
            // (before the quotient is looked at: a residual of 0 makes it 0 / 0)
            if (fin && rho <= stop_rr) {
                done = 1;
                status = kCgConverged;
            } else if (!fin || !pos) {
                done = 1;
                status = kCgBreakdown;
            } else if (iters >= A.max_iters) {
                done = 1;
                status = kCgMaxIter;
            }
        }
        if (done && lane == 0 && bid == 0) {
            A.st->iters = iters;
            A.st->status = status;
            A.st->rr = rho;
            A.st->rr0 = rr0;
            A.st->done = 1;
        }
        return done;
    }
    __device__ __forceinline__ void next(double g, double quot) {
        rz = g;
        ra = rz * __shfl_sync(0xffffffffu, quot, 0);
    }
};
// What a finished run tells the blocks.
enum SoloEnd : int { kSoloRuns = 0, kSoloKeep = 1, kSoloDrop = 2 };

// The block's three sums from its (up to) 16 warp sums, by one warp: product q
// in lanes 8 q .. 8 q + 7 (0 in the last eight).
template <typename T>
__device__ __forceinline__ typename Share<T>::Wide block_shares(const typename Share<T>::type (*red)[16], int nw,
                                                                int lane) {
    using Sh = Share<T>;
    const int q = lane >> 3, k = lane & 7;
    typename Sh::Wide v = Sh::wide(q < 3 ? red[q][k] : Sh::zero());
    if (nw > 8) v = Sh::add(v, Sh::wide(q < 3 ? red[q][k + 8] : Sh::zero()));
    v = Sh::add(v, Sh::shfl(v, 4));
    v = Sh::add(v, Sh::shfl(v, 1));
    return Sh::add(v, Sh::shfl(v, 2));
}

// The loop of the kernel below is kept small on purpose (no unrolling, one copy
// of the star arithmetic): each of its phases runs once per iteration, and
// with 40 KB of loop the instruction fetches took longer than the phases
// (301 x 301 squares: 15k cycles per iteration).
// Measured per iteration, with the kernels it replaces: 301 x 301 squares 4.3 us
// (fused pass 16), 64^3 Kuhn 9.8 (operator, update and halo kernels 25), FP64
// 64 x 64 squares 8.3 (25), FP64 40^3 18 (68).  Bound (cycles of an iteration's
// phases): 301 x 301 squares 3.7k the update, stars and node sums, 2 to 3k the
// scalars (dependent FP64 operations), the rest the exchange (a word from one
// SM's store to another's poll takes 1.7 us on this part); 64^3: 4.6k the stars
// (half their records stream from L2), 4.5k the node sums, 6k the exchange; FP64
// 40^3: 15k of 37k the stars, at the FP64 pipe's rate.
// bid, G: this block's number among the mesh's G blocks.  BATCH: other runs share
// the SMs.  The run's end, or kSoloRuns after a wait's limit.
template <int D, typename T, bool BATCH>
__device__ __forceinline__ int solo_run_block(const SoloArgs<T> &A, const int bid, const int G) {
    extern __shared__ __align__(128) unsigned char smem[];
    constexpr bool F32 = sizeof(T) == 4;
    constexpr int RES = F32 ? kSoloResident : 1;
    constexpr int kW = Tagged<T>::kWords;
    constexpr bool kLanes = F32 && !BATCH;   // one warp reads a product's shares, else 32 at a time
    // (done: set when the run ends, by this thread, and not after a wait's limit)
    if (bid == 0 && threadIdx.x == 0) A.st->done = 0;
    T *val = reinterpret_cast<T *>(smem + A.L.val), *sr = reinterpret_cast<T *>(smem + A.L.r),
      *ss = reinterpret_cast<T *>(smem + A.L.s), *sp = reinterpret_cast<T *>(smem + A.L.p),
      *sx = reinterpret_cast<T *>(smem + A.L.x), *sdi = reinterpret_cast<T *>(smem + A.L.di),
      *sm = reinterpret_cast<T *>(smem + A.L.m), *sw = reinterpret_cast<T *>(smem + A.L.w),
      *contrib = reinterpret_cast<T *>(smem + A.L.contrib);
    uint32_t *goff = reinterpret_cast<uint32_t *>(smem + A.L.goff), *ell = reinterpret_cast<uint32_t *>(smem + A.L.ell);
    int4 *sh = reinterpret_cast<int4 *>(smem + A.L.sh);
    using Sh = Share<T>;
    using ST = typename Sh::type;
    __shared__ ST s_red[3][16];   // warps' sums; entries past the last warp stay 0
    __shared__ typename Sh::Wide s_sum[3][kLanes ? 1 : kSoloMaxBlocks / 32];   // parts of the products' sums
    __shared__ T s_alpha, s_beta;
    __shared__ int s_end;
    const int tid = threadIdx.x, NT = blockDim.x, lane = tid & 31, wid = tid >> 5, nw = NT >> 5;
    const int n_seg = (G + 31) / 32;
    const int ns = F32 ? nw : 4;   // warps that send the block's shares
    const SoloBlock B = A.blocks[bid];
    const int n_sh = B.n_loc - B.n_int;
    // ---- the block's part of the mesh and of the residual
    for (int l = tid; l < B.n_loc; l += NT) {
        const int g = A.gid[B.node0 + l];
        sr[l] = (T)(A.r64[g] * A.scale);
        sdi[l] = A.dinv[g];
        sm[l] = A.mtot[g];
        val[l] = ss[l] = sp[l] = sx[l] = sw[l] = T(0);
    }
    for (int k = tid; k <= (B.n_loc + 31) / 32; k += NT) goff[k] = A.goff[B.goff0 + k];
    for (int k = tid; k < B.n_ell; k += NT) ell[k] = A.ell[B.ell0 + k];
    for (int k = tid; k < n_sh; k += NT) sh[k] = A.sh[B.sh0 + k];
    auto load_star = [&](StarF<D> &S, int q) {
        const int s = B.star0 + q;
        const uint4 id = __ldg(A.ids4 + s);
        const uint32_t id4 = __ldg(A.ids1 + s);
        if (D == 3) S.v[kStarVec<D> - 1] = make_uint4(0u, 0u, 0u, 0u);
        S.load(A.srec + (size_t)(s / kStarLanes) * (A.srows * kStarLanes) + s % kStarLanes);
        S.v[0] = id;
        S.v[1].x = id4;
    };
    auto eval_star = [&](const StarF<D> &S, T *out) {
        if constexpr (F32) {
            const StarIds id = S.ids();
            if (id.nr() == 6) star_eval_nr<D, 6>(S, id, val, out);
            else if (id.nr()) star_eval_any<D>(S, id, val, out);
        }
    };
    StarF<D> res[RES];
    if (F32) {
#pragma unroll
        for (int k = 0; k < RES; ++k) {
            res[k].v[1].x = 0u;
            if (tid + k * NT < B.n_star) load_star(res[k], tid + k * NT);
        }
    }
    SoloScalars<T> sc;
    if (tid < 48) s_red[tid / 16][tid % 16] = Sh::zero();
    if (tid == 0) {
        s_alpha = s_beta = T(0);
        s_end = 0;
        contrib[B.n_star * kPatchSlots] = T(0);   // the lists' padding
    }
    __syncthreads();
    Spin spin;
    for (int it = 0;; ++it) {
        const uint32_t tag = A.tag0 + (uint32_t)it;
        spin.polls = 0;   // (an iteration's words are waited for together)
        if (BATCH && (it & 255) == 255 && bid == 0 && tid == 0) atomicAdd(A.beat, 1u);
        // ---- update
        const T al = s_alpha, be = s_beta;
#pragma unroll 1
        for (int l = tid; l < B.n_loc; l += NT) {
            const T di = sdi[l], r = sr[l];
            const T s2 = fma_rn(be, ss[l], sw[l]);
            const T r2 = fma_rn(-al, s2, r);
            const T p2 = fma_rn(be, sp[l], di * r);
            ss[l] = s2;
            sr[l] = r2;
            sp[l] = p2;
            sx[l] = fma_rn(al, p2, sx[l]);
            val[l] = di * r2;
        }
        __syncthreads();
        // ---- stars
        if constexpr (F32) {
#pragma unroll 1
            for (int q = tid, k = 0; q < B.n_star; q += NT, ++k) {
                StarF<D> S = k == 0 ? res[0] : res[1];
                if (k >= RES) load_star(S, q);
                eval_star(S, contrib + q * kPatchSlots);
            }
        } else {
#pragma unroll 1
            for (int q = tid; q < B.n_star; q += NT) {
                const int s = B.star0 + q;
                const uint4 i4 = __ldg(A.ids4 + s);
                const StarIds id{{i4.x, i4.y, i4.z, i4.w, __ldg(A.ids1 + s)}};
                const double2 *wt =
                    A.sw64 + (size_t)(s / kStarLanes) * (kStarVec64<D> * kStarLanes) + s % kStarLanes;
                T *out = contrib + q * kPatchSlots;
                if (id.nr() == 6) {
                    star_eval64_nr<D, 6>(wt, id, val, out);
                } else if (id.nr()) {
                    StarD<D, 7> S;
                    S.load(wt);
                    star_eval_any<D>(S, id, val, out);
                }
            }
        }
        __syncthreads();
        // ---- node sums and the shares of gamma = r.u, delta = u.A u, rho = r.r
        uint2 *part = (it & 1) ? A.part1 : A.part0;
        typename DotOf<T>::type dg, dd, dr;
#pragma unroll 1
        for (int l = tid; l < B.n_loc; l += NT) {
            T c0 = T(0), c1 = T(0);
#pragma unroll 2
            for (uint32_t o = goff[l >> 5] + lane, e = goff[(l >> 5) + 1]; o < e; o += 32) {
                const uint32_t w = ell[o];
                c0 += contrib[w & 0xffffu];
                c1 += contrib[w >> 16];
            }
            const T c = c0 + c1;
            const T u = val[l], mr = sm[l], r = sr[l];
            T w = fma_rn(fabs(mr), u, c);
            bool own = true;
            if (l < B.n_int) {
                sw[l] = is_dirichlet(mr) ? T(0) : w;
            } else {
                // (a shared unknown's owner carries its row-sum term and its own products)
                const int4 si = sh[l - B.n_int];
                Tagged<T>::put(part, A.n_slots, si.z, c, tag);
                own = si.w != 0;
                if (!own) w = c;
            }
            dd.add_prod(u, w);       // (u = 0 on Dirichlet nodes)
            const T ro = own ? r : T(0);
            dg.add_prod(ro, u);
            dr.add_prod(ro, ro);
        }
        {
            const ST v = warp_share3<T>(Sh::of(dg), Sh::of(dd), Sh::of(dr), lane);
            if ((lane & 7) == 0 && lane < 24) s_red[lane >> 3][wid] = v;
        }
        __syncthreads();
        if (wid < ns) {
            // every block's share to every block: a reader's words lie
            // together and have no other reader (each warp forms the sums)
            const typename Sh::Wide t = block_shares<T>(s_red, nw, lane);
            const int q = lane >> 3, k = lane & 7;
            if (G == 1) {
                if (tid < 24 && k == 0) s_sum[q][0] = t;
            } else if (q < 3) {
                uint4 *exch = A.exch + (size_t)(it & 1) * 3 * G * G + q * G + bid;
                const uint2 b = Sh::bits(t);
#pragma unroll 1
                for (int dst = wid * 8 + k; dst < G; dst += 8 * ns) st_pair(exch + (size_t)3 * dst * G, b.x, b.y, tag);
            }
            __syncwarp();
        }
        if (G > 1) {
            if (kLanes && it > 0) __nanosleep(A.nap);
            // the shared unknowns' partials, which travel beside the shares
#pragma unroll 1
            for (int j = tid; j < n_sh; j += NT) {
                const int l = B.n_int + j;
                const int4 si = sh[j];
                // eight partials' loads are in flight together (a corner of
                // several blocks has that many); one not there yet is polled
                T w = T(0);
#pragma unroll 1
                for (int k0 = si.x; k0 < si.y; k0 += 8) {
                    uint2 f[8 * kW];
#pragma unroll
                    for (int k = 0; k < 8; ++k)
#pragma unroll
                        for (int h = 0; h < kW; ++h) {
                            f[k * kW + h] = make_uint2(0u, tag);
                            if (k0 + k < si.y) f[k * kW + h] = ld_tagged(part + h * A.n_slots + k0 + k);
                        }
                    bool all = true;
#pragma unroll
                    for (int k = 0; k < 8 * kW; ++k) all = all && f[k].y == tag;
                    if (all) {
#pragma unroll
                        for (int k = 0; k < 8; ++k) w += Tagged<T>::of(f + k * kW);
                    } else if (BATCH && it == 0) {
                        int k = 0;   // the first that is not there
#pragma unroll
                        for (int j = 8 * kW - 1; j >= 0; --j)
                            if (f[j].y != tag) k = j;
                        if (spin.again_queued(part + k % kW * A.n_slots + k0 + k / kW, tag, A.beat, A.err)) k0 -= 8;
                    } else if (spin.again(A.spin_limit)) {
                        k0 -= 8;
                    }
                }
                const T mr = sm[l];
                sw[l] = is_dirichlet(mr) ? T(0) : fma_rn(mr, val[l], w);
            }
            if constexpr (!kLanes) {
                // the blocks' shares, 32 of a product to a warp at a time (one
                // warp per product, as below, took the batch 3% longer; FP64 runs
                // 8% shorter on 64 x 64 squares, but with other roundings)
                const uint4 *mine = A.exch + ((size_t)(it & 1) * 3 * G + 3 * bid) * G;
#pragma unroll 1
                for (int sg = wid; sg < 3 * n_seg; sg += nw) {
                    const int q = sg / n_seg, b = (sg - q * n_seg) * 32 + lane;
                    ST v = Sh::zero();
                    if (b < G) {
                        const uint4 *w = mine + q * G + b;
                        uint4 x = ld_pair(w);
                        while ((x.y != tag || x.w != tag) &&
                               (BATCH && it == 0 ? spin.again_queued(reinterpret_cast<const uint2 *>(w) + (x.y == tag),
                                                                     tag, A.beat, A.err)
                                                 : spin.again(A.spin_limit)))
                            x = ld_pair(w);
                        v = Sh::from(x.x, x.z);
                    }
                    __syncwarp();
                    v = Sh::add(v, Sh::shfl(v, 16));
                    v = Sh::add(v, Sh::shfl(v, 8));
                    const typename Sh::Wide t = sum_lanes<T, 8>(Sh::wide(v));
                    if (lane == 0) s_sum[q][sg - q * n_seg] = t;
                }
            } else if (wid < 3) {
                // the blocks' shares, one warp per product: a lane has up to five of
                // them in flight, re-reads those not there yet and adds them in order
                constexpr int kSeg = kSoloMaxBlocks / 32;
                const uint4 *mine = A.exch + ((size_t)(it & 1) * 3 * G + 3 * bid + wid) * G + lane;
                uint4 x[kSeg];
#pragma unroll
                for (int k = 0; k < kSeg; ++k) x[k].y = x[k].w = 32 * k + lane < G ? ~tag : tag, x[k].x = x[k].z = 0u;
                for (;;) {
                    bool all = true;
#pragma unroll
                    for (int k = 0; k < kSeg; ++k)
                        if (x[k].y != tag || x[k].w != tag) x[k] = ld_pair(mine + 32 * k);
#pragma unroll
                    for (int k = 0; k < kSeg; ++k)
                        all = all && x[k].y == tag && x[k].w == tag;
                    if (all || !spin.again(A.spin_limit)) break;
                }
                __syncwarp();
                static_assert(kSeg == 5, "the sum below");
                ST v = Sh::add(Sh::add(Sh::from(x[0].x, x[0].z), Sh::from(x[1].x, x[1].z)),
                               Sh::add(Sh::from(x[2].x, x[2].z), Sh::from(x[3].x, x[3].z)));
                v = Sh::add(v, Sh::from(x[4].x, x[4].z));
                v = Sh::add(v, Sh::shfl(v, 16));
                const typename Sh::Wide t = sum_lanes<T, 16>(Sh::wide(v));
                if (lane == 0) s_sum[wid][0] = t;
            }
        }
        __syncthreads();
        if (wid == 0) {
            // lane 8 q + k: part k of product q
            typename Sh::Wide w = Sh::wide(Sh::zero());
            if constexpr (!kLanes) {   // lane 8 q + k: part k of product q
                const int q = lane >> 3, k = lane & 7;
                if (q < 3 && k < n_seg) w = s_sum[q][k];
                w = sum_lanes<T, 8>(w);
            } else {
                w = s_sum[min(lane >> 3, 2)][0];
            }
            const double v = Sh::total(w);
            const double g = __shfl_sync(0xffffffffu, v, 0), d = __shfl_sync(0xffffffffu, v, 8),
                         rho = __shfl_sync(0xffffffffu, v, 16);
            double quot;
            const int done = sc.advance(A, bid, it, g, d, rho, lane, quot);
            if (lane == 0) {
                s_alpha = (T)quot;
                s_end = !done ? kSoloRuns : sc.status == kCgBreakdown && A.drop ? kSoloDrop : kSoloKeep;
            }
            if (lane == 1 && it > 0) s_beta = (T)quot;
            sc.next(g, quot);
        }
        const bool ok = __syncthreads_and(spin.ok) != 0;
        if (!ok) {
            if (tid == 0) atomicOr(A.err, kErrGridTimeout);
            return kSoloRuns;
        }
        if (s_end) break;
    }
    if (s_end == kSoloDrop) return kSoloDrop;
    for (int l = tid; l < B.n_loc; l += NT)
        if (l < B.n_int || sh[l - B.n_int].w) {
            const int g = A.gid[B.node0 + l];
            A.x64[g] += (double)sx[l] * A.inv_scale;
        }
    return kSoloKeep;
}

template <int D, typename T>
__global__ void __launch_bounds__(512, 1) k_solo_cg(const __grid_constant__ SoloArgs<T> A) {
    solo_run_block<D, T, false>(A, blockIdx.x, gridDim.x);
}

// The same for the meshes of a batch that are in their inner solve.  A thread
// block runs the mesh blocks of its part of the list in order; meshes exchange
// nothing with each other, so a mesh's arithmetic does not depend on the others.
// All lists hold the meshes in one order and all thread blocks are resident, so
// the first unfinished mesh always has its blocks running.
struct SoloJob {
    SoloArgs<float> A;          // (scale, tolerance, cap and tag are the state's)
    BState *bst;
    uint32_t *tag;              // last tag used
    int dim, G;
};
// Two blocks of 256 threads share an SM at 128 registers, so one mesh's exchange
// overlaps the other's arithmetic.  16 meshes, half 2D of up to 167,000
// triangles, half 3D of up to 329,000 tetrahedra: 12.8 ms with a pass over all
// meshes' chunks per iteration, 5.3 here (a 2D mesh of 167,000 triangles takes
// 8 us per iteration beside the others, and it is what the call waits for).
constexpr int kSoloBatchThreads = 256;
__global__ void __launch_bounds__(512, 1) k_solo_batch(const SoloJob *jobs, const int2 *list, const int *ptr) {
    __shared__ __align__(16) SoloJob J;
    __shared__ int s_run;
#pragma unroll 1
    for (int k = ptr[blockIdx.x], e = ptr[blockIdx.x + 1]; k < e; ++k) {
        const int2 me = list[k];            // job, block of the mesh
        __syncthreads();                    // (the previous run's shared memory)
        static_assert(sizeof(SoloJob) % 4 == 0, "word copy");
        for (int w = threadIdx.x; w < (int)(sizeof(SoloJob) / 4); w += blockDim.x)
            reinterpret_cast<uint32_t *>(&J)[w] = reinterpret_cast<const uint32_t *>(jobs + me.x)[w];
        __syncthreads();
        if (threadIdx.x == 0) {
            // (the phase changes at the end of the run, which every block of
            // the mesh takes part in: all have read it by then)
            const BState *st = J.bst;
            s_run = st->phase == kPhSolo;
            J.A.scale = st->scale;
            J.A.inv_scale = 1.0 / st->scale;
            J.A.tol2 = st->in.tol2;
            J.A.max_iters = min(st->in.max_iters, (long long)0x20000000);
            J.A.tag0 = *J.tag + 1u;
        }
        __syncthreads();
        if (!s_run) continue;
        const int end = J.dim == 3 ? solo_run_block<3, float, true>(J.A, me.y, J.G)
                                   : solo_run_block<2, float, true>(J.A, me.y, J.G);
        if (end == kSoloRuns) return;       // a wait gave up: the others' will, those for this thread block too
        if (me.y == 0 && threadIdx.x == 0) {
            BState *st = J.bst;
            const long long iters = st->in.iters;   // (this thread wrote it)
            st->iters_total += iters;
            st->phase = kPhResid;
            *J.tag = J.A.tag0 + (uint32_t)iters + 1u;
            atomicAdd(J.A.beat, 1u);
        }
    }
}

// ---------------------------------------------------------------- host side
static int solo_rc(cudaError_t e) {
    if (e == cudaSuccess) return PS_OK;
    ps_set_last_error(cudaGetErrorString(e));
    return cuda_status(e);
}

template <typename F>
static cudaError_t solo_attr(F *func) {
    int dev = 0, optin = 0;
    cudaError_t e = cudaGetDevice(&dev);
    if (e == cudaSuccess) e = cudaDeviceGetAttribute(&optin, cudaDevAttrMaxSharedMemoryPerBlockOptin, dev);
    cudaFuncAttributes fa;
    if (e == cudaSuccess) e = cudaFuncGetAttributes(&fa, (const void *)func);
    if (e == cudaSuccess)
        e = cudaFuncSetAttribute((const void *)func, cudaFuncAttributeMaxDynamicSharedMemorySize,
                                 optin - (int)fa.sharedSizeBytes);
    return e;
}

int solo_set_attrs() {
    cudaError_t e = solo_attr(k_solo_cg<2, float>);
    if (e == cudaSuccess) e = solo_attr(k_solo_cg<3, float>);
    if (e == cudaSuccess) e = solo_attr(k_solo_cg<2, double>);
    if (e == cudaSuccess) e = solo_attr(k_solo_cg<3, double>);
    if (e == cudaSuccess) e = solo_attr(k_solo_batch);
    return solo_rc(e);
}

// Resident blocks of a kernel on the device.
template <typename F>
static int64_t solo_resident(F *k, int threads, uint32_t bytes, int sms) {
    int per = 0;
    const cudaError_t e = cudaOccupancyMaxActiveBlocksPerMultiprocessor(&per, k, threads, bytes);
    cudaGetLastError();
    return e == cudaSuccess ? (int64_t)per * sms : 0;
}
constexpr uint32_t kSoloSmemMax = 226 * 1024;

// A mesh too large even for its lists alone (a star and its share of a
// block's nodes take over 80 bytes of FP32 shared memory).
static bool solo_too_large(const ps_mesh *m) {
    return m->prep.n_patches * 80 > (int64_t)std::min(m->ctx->sms, kSoloMaxBlocks) * 227 * 1024;
}

// Blocks of about `stars` stars; null: a block's lists exceed 16 bits.
static Solo *solo_sizes(const ps_mesh *m, int stars, SoloPrep &sp) {
    build_solo(m->prep, m->ctx->sms, stars, sp);
    if (sp.max_loc * 4 > 65535 || (int64_t)sp.max_star * kPatchSlots > 65535) return nullptr;
    Solo *S = new Solo();
    S->n_blocks = (int)sp.blocks.size();
    S->n_slots = sp.n_slots;
    S->mean_star = (int)(m->prep.n_patches / std::max(1, S->n_blocks));
    S->sm32 = solo_smem(sp, 4);
    S->sm64 = solo_smem(sp, 8);
    S->threads = sp.max_star <= 128 ? 128 : sp.max_star <= 256 ? 256 : 512;
    return S;
}

// Device copy of a layout into `owner`.  Where the context has no room for it
// the mesh goes without: *ok = false, PS_OK.
static int solo_arrays(ps_mesh *m, const SoloPrep &sp, Solo *S, std::vector<DevAlloc> &owner, bool *ok) {
    const PrepMesh &pm = m->prep;
    std::vector<uint32_t> i4((size_t)pm.patch_total * 4), i1((size_t)pm.patch_total);
    for (int64_t q = 0; q < pm.patch_total; ++q) {
        for (int k = 0; k < 4; ++k) i4[q * 4 + k] = sp.ids[q * kStarIds + k];
        i1[q] = sp.ids[q * kStarIds + 4];
    }
    int rc = PS_OK;
    std::vector<DevAlloc> mine;
    auto up = [&](auto **dst, const void *src, size_t bytes) {
        void *p = nullptr;
        if (rc == PS_OK) rc = dalloc(m->ctx, &p, bytes, mine);
        if (rc == PS_OK && bytes) rc = solo_rc(cudaMemcpy(p, src, bytes, cudaMemcpyHostToDevice));
        *dst = reinterpret_cast<std::remove_reference_t<decltype(*dst)>>(p);
    };
    up(&S->blocks, sp.blocks.data(), sp.blocks.size() * sizeof(SoloBlock));
    up(&S->ids4, i4.data(), i4.size() * 4);
    up(&S->ids1, i1.data(), i1.size() * 4);
    up(&S->gid, sp.gid.data(), sp.gid.size() * 4);
    up(&S->goff, sp.goff.data(), sp.goff.size() * 4);
    up(&S->ell, sp.ell.data(), sp.ell.size() * 4);
    up(&S->sh, sp.sh.data(), sp.sh.size() * 4);
    *ok = rc == PS_OK;
    if (*ok) owner.insert(owner.end(), mine.begin(), mine.end());
    else dfree_all(m->ctx, mine);
    if (rc == PS_ENOMEM) {
        cudaGetLastError();
        rc = PS_OK;
    }
    return rc;
}

int solo_upload(ps_mesh *m) {
    if (solo_too_large(m)) return PS_OK;
    SoloPrep sp;
    Solo *S = solo_sizes(m, kSoloStars, sp);
    if (!S) return PS_OK;
    // one block per SM: cooperative launch needs them all resident
    auto fits = [&](auto *k, uint32_t bytes) {
        return bytes <= kSoloSmemMax && solo_resident(k, S->threads, bytes, m->ctx->sms) >= S->n_blocks;
    };
    const bool d2 = m->prep.dim == 2;
    S->fp32 = d2 ? fits(k_solo_cg<2, float>, S->sm32.total) : fits(k_solo_cg<3, float>, S->sm32.total);
    S->fp64 = d2 ? fits(k_solo_cg<2, double>, S->sm64.total) : fits(k_solo_cg<3, double>, S->sm64.total);
    bool ok = S->fp32 || S->fp64;
    const int rc = ok ? solo_arrays(m, sp, S, m->allocs, &ok) : PS_OK;
    if (ok) m->solo = S;
    else delete S;
    return rc;
}

void solo_release(ps_mesh *m) {
    delete m->solo;
    m->solo = nullptr;
}

// Bytes of the exchanged words: partial sums (two buffers of 8 bytes per FP32
// word) and shares, each from a line of its own (the words of a block that share
// lines with others arrive later: 301 x 301 squares +2.5% per solve).
template <typename T>
static size_t solo_part_bytes(const Solo &S) {
    return ((size_t)std::max(S.n_slots, 1) * 2 * Tagged<T>::kWords * sizeof(uint2) + 255) / 256 * 256;
}
static size_t solo_exch_bytes(const Solo &S) {
    return ((size_t)6 * S.n_blocks * S.n_blocks * sizeof(uint4) + 255) / 256 * 256;
}

bool solo_ready(ps_mesh *m) {
    Solo &S = *m->solo;
    if (S.exch) return true;
    void *p = nullptr;
    if (dalloc(m->ctx, &p, solo_part_bytes<double>(S) + solo_exch_bytes(S), m->ws.allocs) != PS_OK) {
        cudaGetLastError();
        return false;
    }
    S.part = p;
    S.exch = (uint4 *)((char *)p + solo_part_bytes<double>(S));
    S.tag = 0;
    return true;
}

// What a run reads of the mesh, and its exchanged words.
template <typename T>
static SoloArgs<T> solo_args(const ps_mesh *m, const Solo &S, void *part, uint4 *exch) {
    constexpr bool F32 = sizeof(T) == 4;
    SoloArgs<T> A;
    std::memset(&A, 0, sizeof(A));
    A.blocks = S.blocks;
    A.ids4 = S.ids4;
    A.ids1 = S.ids1;
    A.gid = S.gid;
    A.goff = S.goff;
    A.ell = S.ell;
    A.sh = S.sh;
    A.srec = m->dev.srec;
    A.srows = m->dev.srows;
    A.sw64 = m->dev.sw64;
    A.dinv = F32 ? (const T *)m->dev.dinv32 : (const T *)m->dev.dinv64;
    A.mtot = F32 ? (const T *)m->dev.mtot32 : (const T *)m->dev.mtot64;
    A.part0 = (uint2 *)part;
    A.part1 = A.part0 + (size_t)S.n_slots * Tagged<T>::kWords;
    A.n_slots = S.n_slots;
    A.r64 = m->ws.r64;
    A.x64 = m->ws.x64;
    A.relative = F32 ? 1 : 0;
    A.drop = F32 ? 1 : 0;
    A.exch = exch;
    A.st = m->ws.st;
    A.err = m->ctx->d_err;
    A.L = F32 ? S.sm32 : S.sm64;
    return A;
}

// Time between a block's stores and its first poll, in FP32 runs alone on the
// GPU.  A word that is polled before it has arrived was seen about 2 us later than
// one that is not, so the first poll waits as long as the words of this size of
// mesh take.  Iterations in us without / with this wait, and of the code before
// it: 20^3 Kuhn 5.5 / 4.1, 5.1; 28^3 5.9 / 5.3, 5.5; 181 x 181 squares 5.9 / 4.1,
// 5.1; 301 x 301 5.2 (550 ns: 5.7) / 4.3, 5.4; 50^3 6.9 (550 ns: 7.1) / 6.7, 7.0;
// 48 x 48 5.1 (550 ns: 4.7) / 3.5, 3.5.  FP64 runs, whose blocks reach the poll
// later, are up to 3% slower with any.
static uint32_t solo_nap(const Solo &S, int dim) {
    if (S.n_blocks <= 24) return 400;
    return S.mean_star > (dim == 2 ? 150 : 640) ? 250 : 550;
}

template <typename T>
int solo_run(ps_mesh *m, double scale, double tol2, long long max_iters, bool nan_breaks, uint32_t spin_limit,
             cudaStream_t s) {
    constexpr bool F32 = sizeof(T) == 4;
    Solo &S = *m->solo;
    // tags of a run: tag + 1 .. tag + its iterations + 1 (never reused before
    // the words are cleared; a run that gave up leaves tag = 0)
    if (S.tag == 0 || S.tag > 0x40000000u || max_iters > 0x20000000) {
        const cudaError_t e = cudaMemsetAsync(S.part, 0, solo_part_bytes<double>(S) + solo_exch_bytes(S), s);
        if (e != cudaSuccess) return solo_rc(e);
        S.tag = 1;
    }
    SoloArgs<T> A = solo_args<T>(m, S, S.part, S.exch);
    A.scale = scale;
    A.inv_scale = 1.0 / scale;
    A.tol2 = tol2;
    A.nan_breaks = nan_breaks ? 1 : 0;
    A.spin_limit = spin_limit;
    A.nap = solo_nap(S, m->dev.dim);
    A.max_iters = std::min(max_iters, (long long)0x20000000);
    A.tag0 = S.tag + 1;
    cudaLaunchConfig_t cfg;
    std::memset(&cfg, 0, sizeof(cfg));
    cfg.gridDim = dim3(S.n_blocks);
    cfg.blockDim = dim3(F32 ? S.threads : std::min(S.threads, 256));
    cfg.dynamicSmemBytes = A.L.total;
    cfg.stream = s;
    cudaLaunchAttribute attr[1];
    attr[0].id = cudaLaunchAttributeCooperative;
    attr[0].val.cooperative = 1;
    cfg.attrs = attr;
    cfg.numAttrs = 1;
    void *args[] = {&A};
    const void *k = m->dev.dim == 2 ? (const void *)k_solo_cg<2, T> : (const void *)k_solo_cg<3, T>;
    m->launches += 1;
    return solo_rc(cudaLaunchKernelExC(&cfg, k, args));
}
template int solo_run<float>(ps_mesh *, double, double, long long, bool, uint32_t, cudaStream_t);
template int solo_run<double>(ps_mesh *, double, double, long long, bool, uint32_t, cudaStream_t);

// ---------------------------------------------------------------- batches
bool solo_batch_size(const ps_mesh *m) {
    return !solo_too_large(m) && m->prep.n_patches <= (int64_t)std::min(m->ctx->sms, kSoloMaxBlocks) * kSoloBatchStars;
}

int solo_batch_layout(ps_mesh *m, std::vector<DevAlloc> &owner, Solo **out) {
    *out = nullptr;
    if (solo_too_large(m)) return PS_OK;
    if (!solo_batch_size(m)) {
        // every SM either way: the layout of the mesh alone
        if (m->solo && m->solo->fp32 &&
            solo_resident(k_solo_batch, m->solo->threads, m->solo->sm32.total, m->ctx->sms) >= m->solo->n_blocks)
            *out = m->solo;
        return PS_OK;
    }
    SoloPrep sp;
    Solo *S = solo_sizes(m, kSoloBatchStars, sp);
    if (!S) return PS_OK;
    S->threads = kSoloBatchThreads;
    bool ok = S->sm32.total <= kSoloSmemMax &&
              solo_resident(k_solo_batch, kSoloBatchThreads, S->sm32.total, m->ctx->sms) >= S->n_blocks;
    const int rc = ok ? solo_arrays(m, sp, S, owner, &ok) : PS_OK;
    if (ok) *out = S;
    else delete S;
    return rc;
}

int solo_plan_build(BatchPlan &plan, cudaStream_t s) {
    plan.launches.clear();
    // longest runs (iterations ~ nodes per side) first, the larger blocks of
    // the meshes laid out for a solve alone after the others
    std::vector<int> order;
    for (size_t i = 0; i < plan.meshes.size(); ++i)
        if (plan.h_meshes[i].solo) order.push_back((int)i);
    if (order.empty()) return PS_OK;
    auto threads = [&](int i) { return plan.h_meshes[i].solo->threads; };
    auto side = [&](int i) {
        const PrepMesh &p = plan.meshes[i]->prep;
        return std::pow((double)p.n_nodes, 1.0 / p.dim);
    };
    std::stable_sort(order.begin(), order.end(), [&](int a, int b) {
        return threads(a) != threads(b) ? threads(a) < threads(b) : side(a) > side(b);
    });
    std::vector<SoloJob> jobs(order.size());
    std::vector<int2> list;
    std::vector<int> ptr;
    size_t words = 0;
    for (size_t j0 = 0, j1; j0 < order.size(); j0 = j1) {
        SoloLaunch w{(int)ptr.size(), 0, threads(order[j0]), 0u};
        for (j1 = j0; j1 < order.size() && threads(order[j1]) == w.threads; ++j1)
            w.smem = std::max(w.smem, plan.h_meshes[order[j1]].solo->sm32.total);
        const int64_t room = solo_resident(k_solo_batch, w.threads, w.smem, plan.ctx->sms);
        // a mesh takes the thread blocks that are free first
        std::vector<std::vector<int2>> mine(room);
        std::vector<std::pair<double, int>> free(room);   // when, which
        for (int64_t k = 0; k < room; ++k) free[k] = {0.0, (int)k};
        for (size_t j = j0; j < j1; ++j) {
            const Solo &S = *plan.h_meshes[order[j]].solo;
            if (S.n_blocks > room) {
                ps_set_last_error("batch: a mesh's blocks are not resident together");
                return PS_EINVAL;
            }
            std::partial_sort(free.begin(), free.begin() + S.n_blocks, free.end());
            const double end = free[S.n_blocks - 1].first + side(order[j]);
            for (int k = 0; k < S.n_blocks; ++k) {
                mine[free[k].second].push_back(make_int2((int)j, k));
                free[k].first = end;
            }
            words += solo_part_bytes<float>(S) + solo_exch_bytes(S);
        }
        for (const auto &v : mine) {
            if (v.empty()) continue;
            ptr.push_back((int)list.size());
            list.insert(list.end(), v.begin(), v.end());
            w.blocks++;
        }
        ptr.push_back((int)list.size());
        plan.launches.push_back(w);
    }
    // jobs, block lists, then what starts at zero: tags, the beat and words
    auto pad = [](size_t b) { return (b + 255) / 256 * 256; };
    const size_t at_list = pad(jobs.size() * sizeof(SoloJob)), at_ptr = at_list + pad(list.size() * sizeof(int2)),
                 at_tag = at_ptr + pad(ptr.size() * 4), at_words = at_tag + pad((jobs.size() + 1) * 4);
    int rc = plan_buf(plan.ctx, plan.buf_solo, at_words + words);
    if (rc != PS_OK) return rc;
    char *base = (char *)plan.buf_solo.p, *next = base + at_words;
    for (size_t j = 0; j < order.size(); ++j) {
        const ps_mesh *m = plan.meshes[order[j]];
        const Solo &S = *plan.h_meshes[order[j]].solo;
        SoloJob &J = jobs[j];
        std::memset(&J, 0, sizeof(J));
        J.A = solo_args<float>(m, S, next, (uint4 *)(next + solo_part_bytes<float>(S)));
        next += solo_part_bytes<float>(S) + solo_exch_bytes(S);
        J.A.drop = 0;      // (the batch's correction follows a breakdown too)
        J.A.spin_limit = plan.spin_limit;
        J.A.beat = (uint32_t *)(base + at_tag) + jobs.size();
        J.bst = plan.d_st + order[j];
        J.A.st = &J.bst->in;
        J.tag = (uint32_t *)(base + at_tag) + j;
        J.dim = m->dev.dim;
        J.G = S.n_blocks;
    }
    plan.d_jobs = base;
    plan.d_list = (int2 *)(base + at_list);
    plan.d_ptr = (int *)(base + at_ptr);
    plan.zero_at = base + at_tag;
    plan.zero_bytes = at_words + words - at_tag;
    // pageable sources: staged by the runtime before the calls return
    rc = solo_rc(cudaMemcpyAsync(base, jobs.data(), jobs.size() * sizeof(SoloJob), cudaMemcpyHostToDevice, s));
    if (rc == PS_OK)
        rc = solo_rc(cudaMemcpyAsync(plan.d_list, list.data(), list.size() * sizeof(int2), cudaMemcpyHostToDevice, s));
    if (rc == PS_OK) rc = solo_rc(cudaMemcpyAsync(plan.d_ptr, ptr.data(), ptr.size() * 4, cudaMemcpyHostToDevice, s));
    return rc == PS_OK ? solo_plan_clear(plan, s) : rc;
}

int solo_plan_clear(BatchPlan &plan, cudaStream_t s) {
    plan.tag_high = 0;
    if (plan.launches.empty()) return PS_OK;
    return solo_rc(cudaMemsetAsync(plan.zero_at, 0, plan.zero_bytes, s));
}

int solo_plan_enqueue(BatchPlan &plan, cudaStream_t s) {
    for (const SoloLaunch &w : plan.launches) {
        cudaLaunchConfig_t cfg;
        std::memset(&cfg, 0, sizeof(cfg));
        cfg.gridDim = dim3(w.blocks);
        cfg.blockDim = dim3(w.threads);
        cfg.dynamicSmemBytes = w.smem;
        cfg.stream = s;
        cudaLaunchAttribute attr[1];
        attr[0].id = cudaLaunchAttributeCooperative;
        attr[0].val.cooperative = 1;
        cfg.attrs = attr;
        cfg.numAttrs = 1;
        const SoloJob *jobs = (const SoloJob *)plan.d_jobs;
        const int2 *list = plan.d_list;
        const int *ptr = plan.d_ptr + w.first;
        void *args[] = {&jobs, &list, &ptr};
        const int rc = solo_rc(cudaLaunchKernelExC(&cfg, (const void *)k_solo_batch, args));
        if (rc != PS_OK) return rc;
    }
    return PS_OK;
}

}  // namespace ps
