// Chunked matrix-free P1 operator and the fused CG kernels.
//
// One thread block processes one chunk (layout.h):
//   1. one elected thread moves the chunk's incidence pointers and lists into
//      shared memory with bulk copies signalled on an mbarrier;
//   2. the block gathers the input vector for its local nodes (contiguous for
//      interior nodes, through the shared-node ids otherwise), masking
//      Dirichlet nodes; in CG mode it forms the new search direction
//      p = D^-1 r + beta p on the fly and stores it for its interior nodes;
//   3. one thread per star patch forms the patch's contributions to its nodes
//      in shared memory, from the patch's record and weights (read coalesced
//      from global memory: nothing of them is staged);
//   4. one thread per local node sums its contributions in incidence-list
//      order, adds the row-sum term and writes its row (interior node) or a
//      partial sum (shared node).
// A second kernel adds the partial sums of shared nodes in a fixed order.
// Dot products are accumulated in FP64 per block and reduced by the last
// block to finish, in a fixed order, so every result is bitwise reproducible.
#pragma once
#include "device.cuh"

namespace ps {

enum Mode : int { kApply = 0, kResid = 2, kDiag = 3 };

struct SmemLayout {
    uint32_t val, aux, incp, inc, contrib, red, bar, total;
};

// Shared memory of k_cg2_stars (cg2s.cuh): the chunk's records, its incidence
// pointers and lists, node values.
struct StarSmem {
    uint32_t rec, incp, inc, val, bar, total;
};

struct MeshDev {
    int dim, n_chunks;
    int64_t n_nodes, n_int, n_shared, n_pad;
    const ChunkDesc *chunks;
    const uint4 *srec;       // star records: ids and FP32 weights (layout.h)
    int srows;               // rows per record
    int stream;              // 1: the records exceed what L2 keeps from one pass to the next
    const uint16_t *inc_rec; // incidence lists of k_cg2_stars (null: not used): contributions in the records' place
    const double2 *sw64;     // FP64 star weights
    const float *mrow32;     // [loc_total] row sums of the chunk's patches, sign bit set on Dirichlet nodes
    const double *mrow64;
    const float *mtot32;     // [n_pad] the same summed over all chunks, per unknown
    const double *mtot64;
    const uint16_t *incp, *inc;
    const int32_t *sh_ids, *shr_ptr, *sh_dest;
    const int4 *sh_info;     // [sh_total] node id, partial range [begin, end), owner flag
    const float *dinv32;
    const double *dinv64;
    // what the weights are formed from (k_star_build)
    const double *geo64;     // [patch_total * kPatchMax * kGeoWords<dim>] element geometry
    const double *bdt2_64;   // [patch_total * kPatchMax] beta*dt^2 per element slot
    const double *alpha64;   // [loc_total] alpha of the local nodes, sign bit set on Dirichlet nodes
    const uint8_t *dirichlet;
    int *err;
    int lumped;              // 1: mass term by vertex quadrature (mass-lumped variant)
    SmemLayout sm32, sm64;
    StarSmem sms;
};

// Scalars of one CG run, kept on the device.
struct CgState {
    double rz, pq, alpha, beta, rr, rr0, stop_rr, bb;
    long long iters, max_iters;
    int done, status;
    unsigned int cnt_a, cnt_b;
    int first, free_run;     // fused engine: first = the start pass is next;
                             // free_run = never stop (kernel timing only)
    double tol2;             // fused engine: relative stopping tolerance squared
};

enum CgStatus : int { kCgRunning = 0, kCgConverged = 1, kCgMaxIter = 2, kCgBreakdown = 3 };

template <typename T>
struct VecArgs {
    const T *x;      // apply / resid: input vector
    T *y;            // apply: output; resid: r
    const T *b;      // resid: right-hand side (0 on Dirichlet nodes)
    T *partial;      // [sh_total] partial sums of shared local nodes
    double *dotbuf;  // resid: per-block dot partials
    CgState *st;     // resid: receives r.r
    // apply in the caller's numbering (null: x and y in the internal one): the
    // caller's vertex of every local node and of every unknown, and the
    // vertices merged into an unknown
    const int32_t *loc_user, *old_of_new, *slave_ptr, *slave;
};

__device__ __forceinline__ float cg_dir(float dinv, float r, float beta, float p) {
    return __fmaf_rn(beta, p, __fmul_rn(dinv, r));
}
__device__ __forceinline__ double cg_dir(double dinv, double r, double beta, double p) {
    return __fma_rn(beta, p, __dmul_rn(dinv, r));
}

__device__ __forceinline__ int ld_flag(const int *p) { return *(volatile const int *)p; }

// Shared-memory view of one chunk.
template <typename T>
struct ChunkSmem {
    T *val, *aux, *contrib;
    uint16_t *incp, *inc;
    uint64_t *bar;
    double *red;
};

template <typename T>
__device__ __forceinline__ ChunkSmem<T> chunk_smem(unsigned char *smem, const SmemLayout &L) {
    ChunkSmem<T> S;
    S.val = reinterpret_cast<T *>(smem + L.val);
    S.aux = reinterpret_cast<T *>(smem + L.aux);
    S.contrib = reinterpret_cast<T *>(smem + L.contrib);
    S.incp = reinterpret_cast<uint16_t *>(smem + L.incp);
    S.inc = reinterpret_cast<uint16_t *>(smem + L.inc);
    S.bar = reinterpret_cast<uint64_t *>(smem + L.bar);
    S.red = reinterpret_cast<double *>(smem + L.red);
    return S;
}

// Row 0 of patch q of a chunk (kStarLanes patches per group).
template <int D>
__device__ __forceinline__ const uint4 *star_rec(const MeshDev &m, const ChunkDesc &cd, int q) {
    return m.srec + (size_t)((cd.patch_off + q) / kStarLanes) * (m.srows * kStarLanes) + q % kStarLanes;
}
template <int D>
__device__ __forceinline__ const double2 *star_wt64(const MeshDev &m, const ChunkDesc &cd, int q) {
    return m.sw64 + (size_t)((cd.patch_off + q) / kStarLanes) * (kStarVec64<D> * kStarLanes) + q % kStarLanes;
}
template <typename T>
__device__ __forceinline__ const T *chunk_mrow(const MeshDev &m, const ChunkDesc &cd) {
    return (sizeof(T) == 4 ? reinterpret_cast<const T *>(m.mrow32) : reinterpret_cast<const T *>(m.mrow64)) +
           cd.node_off;
}

// Thread 0 issues the bulk copies of chunk cd's incidence pointers and lists.
// When the shared memory was used by an earlier chunk, the caller has
// synchronised the block; the proxy fence orders those generic-proxy reads
// before the async-proxy writes.
template <typename T>
__device__ __forceinline__ void stage_issue(const MeshDev &m, const ChunkDesc &cd, const ChunkSmem<T> &S) {
    if (threadIdx.x != 0) return;
    const uint32_t b_incp = (uint32_t)((cd.n_loc + 1 + kIncpPad - 1) / kIncpPad * kIncpPad) * 2u;
    const uint32_t b_inc = (uint32_t)((cd.n_inc + kIncPad - 1) / kIncPad * kIncPad) * 2u;
    fence_proxy_async_smem();
    mbar_arrive_expect_tx(S.bar, b_incp + b_inc);
    bulk_g2s(S.incp, m.incp + cd.incp_off, b_incp, S.bar);
    bulk_g2s(S.inc, m.inc + cd.inc_off, b_inc, S.bar);
}

// Wait for the staged data (bounded); block-uniform result.  On timeout the
// error flag is set and the copies in flight are waited for once more.
template <typename T>
__device__ __forceinline__ bool stage_wait(const MeshDev &m, const ChunkSmem<T> &S, uint32_t &phase) {
    bool ok = mbar_wait_bounded(S.bar, phase);
    ok = __syncthreads_and(ok);
    if (!ok) {
        if (threadIdx.x == 0) atomicOr(m.err, kErrMbarTimeout);
        mbar_wait_bounded(S.bar, phase);
    }
    phase ^= 1u;
    return ok;
}

// Contributions of every star patch of the chunk into S.contrib; ends with a
// block barrier.  FP32: a thread's first patch may have been loaded earlier
// (PRE: before the gather, so that its record arrives while the gather waits).
template <int D, bool PRE>
__device__ __forceinline__ void stars_eval(const MeshDev &m, const ChunkDesc &cd, const ChunkSmem<float> &S,
                                           const StarF<D> &pre) {
    int q = threadIdx.x;
    if (PRE && q < cd.n_patch) {
        star_eval<D>(pre, S.val, S.contrib + q * kPatchSlots);
        q += blockDim.x;
    }
    for (; q < cd.n_patch; q += blockDim.x) {
        StarF<D> st;
        st.load(star_rec<D>(m, cd, q));
        star_eval<D>(st, S.val, S.contrib + q * kPatchSlots);
    }
    __syncthreads();
}
template <int D, bool PRE>
__device__ __forceinline__ void stars_eval(const MeshDev &m, const ChunkDesc &cd, const ChunkSmem<double> &S,
                                           const StarF<D> &) {
    for (int q = threadIdx.x; q < cd.n_patch; q += blockDim.x)
        star_eval64<D>(star_ids(star_rec<D>(m, cd, q)), star_wt64<D>(m, cd, q), S.val, S.contrib + q * kPatchSlots);
    __syncthreads();
}
template <int D>
__device__ __forceinline__ void star_prefetch(const MeshDev &m, const ChunkDesc &cd, StarF<D> &pre) {
    if ((int)threadIdx.x < cd.n_patch) pre.load(star_rec<D>(m, cd, threadIdx.x));
}

// Sum of contributions c[inc[k]], k in [b, e): four independent partial sums
// in a fixed pattern (deterministic).
template <typename T>
__device__ __forceinline__ T list_sum(const T *__restrict__ c, const uint16_t *__restrict__ inc, int b, int e) {
    T s0 = T(0), s1 = T(0), s2 = T(0), s3 = T(0);
    int k = b;
    for (; k + 3 < e; k += 4) {
        s0 += c[inc[k]];
        s1 += c[inc[k + 1]];
        s2 += c[inc[k + 2]];
        s3 += c[inc[k + 3]];
    }
    for (; k < e; ++k) s0 += c[inc[k]];
    return (s0 + s1) + (s2 + s3);
}
// Sum of the contributions of local node l in incidence order.
template <typename T>
__device__ __forceinline__ T node_sum(const ChunkSmem<T> &S, int l) {
    return list_sum(S.contrib, S.inc, S.incp[l], S.incp[l + 1]);
}

// Process chunk c (apply, residual).  Returns this thread's share of the
// residual's r.r over interior nodes.  `phase` is the mbarrier parity to wait
// for; it flips on return.  Block-uniform; contains __syncthreads.
template <int D, typename T, int MODE>
__device__ typename DotOf<T>::type process_chunk(const MeshDev &m, const VecArgs<T> &a, int c, unsigned char *smem,
                                                 const SmemLayout &L, uint32_t &phase, bool &failed) {
    using Acc = typename DotOf<T>::type;
    constexpr bool kPre = sizeof(T) == 4;
    const ChunkDesc cd = m.chunks[c];
    const ChunkSmem<T> S = chunk_smem<T>(smem, L);
    const int n_loc = cd.n_loc, n_int = cd.n_int;
    stage_issue<T>(m, cd, S);
    const T *mrow = chunk_mrow<T>(m, cd);
    StarF<D> pre;
    if (kPre) star_prefetch<D>(m, cd, pre);
    // ---- gather the input vector (masked on Dirichlet nodes).  The element
    // phase of a chunk whose input is zero on all its nodes (a zero first
    // guess, a zero correction) is skipped: every contribution is then 0.
    bool nonzero = false;
    for (int l0 = threadIdx.x; l0 < n_loc; l0 += 4 * blockDim.x) {
        T v[4], mr[4];
#pragma unroll
        for (int k = 0; k < 4; ++k) {
            const int l = l0 + k * blockDim.x;
            v[k] = mr[k] = T(0);
            if (l < n_loc) {
                const int g = MODE == kApply && a.loc_user ? a.loc_user[cd.node_off + l]
                              : l < n_int                  ? cd.int_begin + l
                                                           : m.sh_ids[cd.sh_off + (l - n_int)];
                v[k] = a.x[g];
                mr[k] = mrow[l];
            }
        }
#pragma unroll
        for (int k = 0; k < 4; ++k) {
            const int l = l0 + k * blockDim.x;
            if (l < n_loc) {
                if (is_dirichlet(mr[k])) v[k] = T(0);
                S.val[l] = v[k];
                nonzero |= v[k] != T(0);
            }
        }
    }
    if (!stage_wait<T>(m, S, phase)) {
        failed = true;
        return Acc();
    }
    const bool work = __syncthreads_or(nonzero) != 0;
    if (work) stars_eval<D, kPre>(m, cd, S, pre);

    // ---- per-node sums in incidence order
    Acc dot;
    for (int l = threadIdx.x; l < n_loc; l += blockDim.x) {
        const T mr = mrow[l];
        T s = work ? fma(fabs(mr), S.val[l], node_sum(S, l)) : T(0);
        const bool dir = is_dirichlet(mr);
        if (dir) s = T(0);
        if (l < n_int) {
            const int g = cd.int_begin + l;
            if (MODE == kApply) {
                a.y[a.loc_user ? a.loc_user[cd.node_off + l] : g] = s;
            } else {
                const T rv = dir ? T(0) : a.b[g] - s;
                a.y[g] = rv;
                dot.add_prod(rv, rv);
            }
        } else {
            a.partial[m.sh_dest[cd.sh_off + (l - n_int)]] = s;
        }
    }
    return dot;
}

// Kernel 1 of an apply or residual: one block per chunk.
template <int D, typename T, int MODE>
__global__ void __launch_bounds__(256) k_chunks(MeshDev m, VecArgs<T> a) {
    extern __shared__ __align__(128) unsigned char smem[];
    const SmemLayout &L = (sizeof(T) == 4) ? m.sm32 : m.sm64;
    uint64_t *s_bar = reinterpret_cast<uint64_t *>(smem + L.bar);
    double *s_red = reinterpret_cast<double *>(smem + L.red);
    grid_dep_launch();   // (k_shared's blocks may start once every block here has)
    if (threadIdx.x == 0) {
        mbar_init(s_bar, 1);
        fence_mbar_init();
    }
    __syncthreads();
    uint32_t phase = 0;
    bool failed = false;
    const typename DotOf<T>::type acc = process_chunk<D, T, MODE>(m, a, blockIdx.x, smem, L, phase, failed);
    if (MODE == kResid) {
        const double dot = block_sum(acc, s_red);
        if (threadIdx.x == 0) a.dotbuf[blockIdx.x] = dot;
    }
}

// Star weights, row sums and the Jacobi diagonal from the mesh's geometry,
// alpha and beta*dt^2, one block per chunk.  beta (may be null): the caller's
// element values, stored as beta*dt^2 per element slot on the way; null: the
// stored ones.  Row by row the diagonal is D_ii = m_i - sum_j A_ij.  Interior
// rows are stored here (0 on Dirichlet rows), shared ones as partial sums
// (k_shared<double, kDiag>), the diagonal's n_part of them and then the row
// sums' (per unknown).  A pass of the FP64 pipe (about 29 operations
// per tetrahedron) that reads 64 bytes per tetrahedron.
template <int D>
__global__ void __launch_bounds__(256, 3) k_star_build(MeshDev m, const int32_t *__restrict__ elem_src,
                                                    const double *__restrict__ beta, double dt2, double *partial,
                                                    int64_t n_part) {
    extern __shared__ __align__(128) unsigned char smem[];
    const ChunkSmem<double> S = chunk_smem<double>(smem, m.sm64);
    if (threadIdx.x == 0) {
        mbar_init(S.bar, 1);
        fence_mbar_init();
    }
    __syncthreads();
    const ChunkDesc cd = m.chunks[blockIdx.x];
    stage_issue<double>(m, cd, S);
    for (int l = threadIdx.x; l < cd.n_loc; l += blockDim.x) S.val[l] = m.alpha64[cd.node_off + l];
    uint32_t phase = 0;
    if (!stage_wait<double>(m, S, phase)) return;   // also the barrier for S.val
    auto w32 = [&](int q) { return reinterpret_cast<float *>(const_cast<uint4 *>(star_rec<D>(m, cd, q))); };
    auto w64 = [&](int q) { return reinterpret_cast<double *>(const_cast<double2 *>(star_wt64<D>(m, cd, q))); };
    double *bdt2 = const_cast<double *>(m.bdt2_64) + (size_t)cd.patch_off * kPatchMax;
    const int32_t *src = elem_src + (size_t)cd.patch_off * kPatchMax;
    for (int q = threadIdx.x; q < cd.n_patch; q += blockDim.x) {
        const StarIds id = star_ids(star_rec<D>(m, cd, q));
        const double *geo = m.geo64 +
                            (size_t)((cd.patch_off + q) / kStarLanes) * (kPatchMax * kGeoWords<D> * kStarLanes) +
                            q % kStarLanes;
        double bd[kPatchMax];
        double2 *b2 = reinterpret_cast<double2 *>(bdt2 + q * kPatchMax);
        if (beta) {
            const int2 *s2 = reinterpret_cast<const int2 *>(src + q * kPatchMax);
#pragma unroll
            for (int j = 0; j < kPatchMax / 2; ++j) {
                const int2 e = __ldg(s2 + j);
                bd[2 * j] = e.x >= 0 ? __ldg(beta + e.x) * dt2 : 0.0;
                bd[2 * j + 1] = e.y >= 0 ? __ldg(beta + e.y) * dt2 : 0.0;
                b2[j] = make_double2(bd[2 * j], bd[2 * j + 1]);
            }
        } else {
#pragma unroll
            for (int j = 0; j < kPatchMax / 2; ++j) {
                const double2 v = b2[j];
                bd[2 * j] = v.x;
                bd[2 * j + 1] = v.y;
            }
        }
        star_build<D>(id, geo, bd, S.val, m.lumped != 0, w32(q), w64(q), S.contrib + q * kPatchSlots);
    }
    __syncthreads();
    for (int l = threadIdx.x; l < cd.n_loc; l += blockDim.x) {
        double ml = node_sum(S, l);
        S.aux[l] = ml;
        if (is_dirichlet(S.val[l])) ml = __longlong_as_double(__double_as_longlong(ml) | (long long)0x8000000000000000ULL);
        const_cast<double *>(m.mrow64)[cd.node_off + l] = ml;
        const_cast<float *>(m.mrow32)[cd.node_off + l] = (float)ml;
        if (l < cd.n_int) {
            const_cast<double *>(m.mtot64)[cd.int_begin + l] = ml;
            const_cast<float *>(m.mtot32)[cd.int_begin + l] = (float)ml;
        } else {
            partial[n_part + m.sh_dest[cd.sh_off + (l - cd.n_int)]] = fabs(ml);
        }
    }
    __syncthreads();
    // off-diagonal row sums, from the weights this thread just stored
    for (int q = threadIdx.x; q < cd.n_patch; q += blockDim.x) {
        const int nr = star_ids(star_rec<D>(m, cd, q)).nr();
        const double *wq = w64(q);
        auto w = [&](int k) { return wq[(k / 2) * 2 * kStarLanes + k % 2]; };
        double *out = S.contrib + q * kPatchSlots;
        double sa = 0.0, sb = 0.0;
        if (D == 3) sa = sb = w(0);
        const double wrap = w(D == 3 ? 1 : 0);
        double prev = wrap;
#pragma unroll
        for (int j = 0; j < kStarRing; ++j) {
            if (j >= nr) break;
            const int k = j == 0 ? (D == 3 ? 2 : 1) : (D == 3 ? 4 : 2) + D * (j - 1);
            const double next = j + 1 < nr ? w((D == 3 ? 4 : 2) + D * j + D - 1) : wrap;
            double o = prev + next + w(k);
            sa += w(k);
            if (D == 3) {
                sb += w(k + 1);
                o += w(k + 1);
            }
            out[2 + j] = o;
            prev = next;
        }
        out[0] = sa;
        if (D == 3) out[1] = sb;
    }
    __syncthreads();
    for (int l = threadIdx.x; l < cd.n_loc; l += blockDim.x) {
        const double d = S.aux[l] - node_sum(S, l);
        if (l < cd.n_int) {
            const double dv = is_dirichlet(S.val[l]) ? 0.0 : 1.0 / d;
            const_cast<double *>(m.dinv64)[cd.int_begin + l] = dv;
            const_cast<float *>(m.dinv32)[cd.int_begin + l] = (float)dv;
        } else {
            partial[m.sh_dest[cd.sh_off + (l - cd.n_int)]] = d;
        }
    }
}

// Kernel 2: shared nodes sum their partials in slot order.  Residual: the
// last block to finish also reduces all dot partials (kernel 1's n_first
// blocks, then this kernel's blocks) into the state's rr.
template <typename T, int MODE>
__global__ void __launch_bounds__(256) k_shared(MeshDev m, VecArgs<T> a, int n_first) {
    __shared__ double s_red[34];
    __shared__ bool s_last;
    typename DotOf<T>::type acc;
    int64_t s = (int64_t)blockIdx.x * blockDim.x + threadIdx.x;
    int kb = 0, ke = 0;
    if (s < m.n_shared) {
        kb = m.shr_ptr[s];
        ke = m.shr_ptr[s + 1];
    }
    grid_dep_wait();     // kernel 1 has ended: its partial sums are there
    for (; s < m.n_shared; s += (int64_t)gridDim.x * blockDim.x) {
        const int64_t g = m.n_int + s;
        T sum = T(0);
        if (s >= (int64_t)gridDim.x * blockDim.x) {
            kb = m.shr_ptr[s];
            ke = m.shr_ptr[s + 1];
        }
        for (int k = kb; k < ke; ++k) sum += a.partial[k];
        const bool dir = m.dirichlet[g] != 0;
        if (MODE == kApply) {
            const T v = dir ? T(0) : sum;
            a.y[a.old_of_new ? a.old_of_new[g] : g] = v;
            if (a.slave_ptr)
                for (int k = a.slave_ptr[g]; k < a.slave_ptr[g + 1]; ++k) a.y[a.slave[k]] = v;
        } else if (MODE == kResid) {
            const T rv = dir ? T(0) : a.b[g] - sum;
            a.y[g] = rv;
            acc.add_prod(rv, rv);
        } else {
            const double dv = dir ? 0.0 : 1.0 / (double)sum;
            const_cast<double *>(m.dinv64)[g] = dv;
            const_cast<float *>(m.dinv32)[g] = (float)dv;
            // the row sums' partials follow the diagonal's (n_first slots)
            double mt = 0.0;
            for (int k = kb; k < ke; ++k) mt += (double)a.partial[n_first + k];
            if (dir) mt = __longlong_as_double(__double_as_longlong(mt) | (long long)0x8000000000000000ULL);
            const_cast<double *>(m.mtot64)[g] = mt;
            const_cast<float *>(m.mtot32)[g] = (float)mt;
        }
    }
    if (MODE != kResid) return;
    const double dot = block_sum(acc, s_red);
    if (threadIdx.x == 0) {
        a.dotbuf[n_first + blockIdx.x] = dot;
        const unsigned int t = atomic_add_acq_rel(&a.st->cnt_a, 1u);
        s_last = (t == gridDim.x - 1);
    }
    __syncthreads();
    if (!s_last) return;
    const double tot = block_sum_array(a.dotbuf, n_first + gridDim.x, s_red);
    if (threadIdx.x == 0) {
        a.st->cnt_a = 0;
        a.st->rr = tot;
    }
}

// Start of an inner FP32 solve of A d = r64 * scale (mixed mode), or of an
// FP64 PCG run from a residual already in r (mode FP64: rsrc == nullptr).
// Sets d = 0, p = 0, rz = r.D^-1 r, rr0 = r.r, stop_rr = tol2 * (rr0 or bb).
template <typename T>
__global__ void __launch_bounds__(256) k_cg_start(int64_t n_pad, const double *__restrict__ rsrc, double scale,
                                                  T *__restrict__ r, T *__restrict__ d, T *__restrict__ p,
                                                  const T *__restrict__ dinv, CgState *st, double *dotbuf,
                                                  double tol2, int relative, long long max_iters) {
    __shared__ double s_red[34];
    __shared__ bool s_last;
    typename DotOf<T>::type arz, arr;
    for (int64_t i = (int64_t)blockIdx.x * blockDim.x + threadIdx.x; i < n_pad; i += (int64_t)gridDim.x * blockDim.x) {
        T ri = rsrc ? (T)(rsrc[i] * scale) : r[i];
        if (rsrc) r[i] = ri;
        if (d) d[i] = T(0);
        p[i] = T(0);
        arz.add_prod(ri, dinv[i] * ri);
        arr.add_prod(ri, ri);
    }
    const double rz = block_sum(arz, s_red);
    const double rr = block_sum(arr, s_red);
    if (threadIdx.x == 0) {
        dotbuf[blockIdx.x] = rz;
        dotbuf[gridDim.x + blockIdx.x] = rr;
        const unsigned int t = atomic_add_acq_rel(&st->cnt_b, 1u);
        s_last = (t == gridDim.x - 1);
    }
    __syncthreads();
    if (!s_last) return;
    const double rz0 = block_sum_array(dotbuf, gridDim.x, s_red);
    const double rr0 = block_sum_array(dotbuf + gridDim.x, gridDim.x, s_red);
    if (threadIdx.x == 0) {
        st->cnt_b = 0;
        st->cnt_a = 0;
        st->rz = rz0;
        st->rr0 = rr0;
        st->rr = rr0;
        st->beta = 0.0;
        st->alpha = 0.0;
        st->iters = 0;
        st->max_iters = max_iters;
        st->stop_rr = relative ? tol2 * rr0 : tol2;
        st->status = kCgRunning;
        st->done = 0;
        if (!isfinite(rz0) || !isfinite(rr0)) {
            st->status = kCgBreakdown;
            st->done = 1;
        } else if (rr0 <= st->stop_rr || rr0 == 0.0) {
            st->status = kCgConverged;
            st->done = 1;
        }
    }
}

// x64 += d32 / scale (mixed-mode correction), vectors padded to 4.
static __global__ void k_correct(int64_t n_pad, double *__restrict__ x, const float *__restrict__ d, double inv_scale) {
    for (int64_t i = (int64_t)blockIdx.x * blockDim.x + threadIdx.x; i < n_pad; i += (int64_t)gridDim.x * blockDim.x)
        x[i] += (double)d[i] * inv_scale;
}

// out_new[i] = in_old[old_of_new[i]] (0 on Dirichlet nodes); element types converted.
template <typename TI, typename TO>
__global__ void k_perm_in(int64_t n, const TI *__restrict__ in, TO *__restrict__ out, const int32_t *__restrict__ old_of_new,
                          const uint8_t *__restrict__ dirichlet) {
    for (int64_t i = (int64_t)blockIdx.x * blockDim.x + threadIdx.x; i < n; i += (int64_t)gridDim.x * blockDim.x)
        out[i] = dirichlet[i] ? TO(0) : (TO)in[old_of_new[i]];
}
// Merged periodic vertices: out[g] += sum of in[v] over the vertices merged
// into unknown g (ascending vertex id; 0 stays on Dirichlet unknowns).
static __global__ void k_add_slaves(int64_t n, const int32_t *__restrict__ ptr, const int32_t *__restrict__ slave,
                                    const double *__restrict__ in, double *__restrict__ out,
                                    const uint8_t *__restrict__ dirichlet) {
    for (int64_t g = (int64_t)blockIdx.x * blockDim.x + threadIdx.x; g < n; g += (int64_t)gridDim.x * blockDim.x) {
        if (dirichlet[g] || ptr[g] == ptr[g + 1]) continue;
        double v = out[g];
        for (int k = ptr[g]; k < ptr[g + 1]; ++k) v += in[slave[k]];
        out[g] = v;
    }
}
// out_old[j] = in_new[new_of_old[j]]
template <typename TI, typename TO>
__global__ void k_perm_out(int64_t n, const TI *__restrict__ in, TO *__restrict__ out, const int32_t *__restrict__ new_of_old) {
    for (int64_t j = (int64_t)blockIdx.x * blockDim.x + threadIdx.x; j < n; j += (int64_t)gridDim.x * blockDim.x)
        out[j] = (TO)in[new_of_old[j]];
}

__device__ __forceinline__ void put_alpha(const MeshDev &m, int64_t k, double a, bool dir) {
    if (dir) a = __longlong_as_double(__double_as_longlong(a) | (long long)0x8000000000000000ULL);
    const_cast<double *>(m.alpha64)[k] = a;
}

// Fill the alpha of every local node: +alpha, or -alpha (sign bit set, also
// for alpha = 0) on Dirichlet nodes.
static __global__ void k_set_alpha(MeshDev m, int64_t n_loc, const int32_t *__restrict__ loc_node,
                                   const double *__restrict__ alpha_new) {
    for (int64_t k = (int64_t)blockIdx.x * blockDim.x + threadIdx.x; k < n_loc; k += (int64_t)gridDim.x * blockDim.x) {
        const int g = loc_node[k];
        put_alpha(m, k, alpha_new[g], m.dirichlet[g] != 0);
    }
}

// The same from caller-numbered alpha: unknown g takes alpha of its master
// vertex old_of_new[g].  wl (may be null, lumped mass): the lumped weight
// |T|/(d+1) summed over the chunk's elements around each local node (wl_tot:
// over all elements, per unknown); alpha then scales it into the row sums, all that a lumped operator takes from it.
static __global__ void k_set_alpha_user(MeshDev m, int64_t n_loc, const int32_t *__restrict__ loc_node,
                                        const int32_t *__restrict__ old_of_new, const double *__restrict__ alpha_user,
                                        const double *__restrict__ wl, const double *__restrict__ wl_tot) {
    if (wl)
        for (int64_t g = (int64_t)blockIdx.x * blockDim.x + threadIdx.x; g < m.n_nodes;
             g += (int64_t)gridDim.x * blockDim.x) {
            double mt = alpha_user[old_of_new[g]] * wl_tot[g];
            if (m.dirichlet[g]) mt = __longlong_as_double(__double_as_longlong(mt) | (long long)0x8000000000000000ULL);
            const_cast<double *>(m.mtot64)[g] = mt;
            const_cast<float *>(m.mtot32)[g] = (float)mt;
        }
    for (int64_t k = (int64_t)blockIdx.x * blockDim.x + threadIdx.x; k < n_loc; k += (int64_t)gridDim.x * blockDim.x) {
        const int g = loc_node[k];
        const double a = alpha_user[old_of_new[g]];
        put_alpha(m, k, a, m.dirichlet[g] != 0);
        if (wl) {
            double ml = a * wl[k];
            if (m.dirichlet[g]) ml = __longlong_as_double(__double_as_longlong(ml) | (long long)0x8000000000000000ULL);
            const_cast<double *>(m.mrow64)[k] = ml;
            const_cast<float *>(m.mrow32)[k] = (float)ml;
        }
    }
}

// bdt2[k] = beta[elem_src[k]] * dt2 (0 on padding slots).
static __global__ void k_set_beta(int64_t n, const int32_t *__restrict__ elem_src, const double *__restrict__ beta,
                                  double dt2, double *b64) {
    for (int64_t k = (int64_t)blockIdx.x * blockDim.x + threadIdx.x; k < n; k += (int64_t)gridDim.x * blockDim.x) {
        const int e = elem_src[k];
        b64[k] = e >= 0 ? beta[e] * dt2 : 0.0;
    }
}

}  // namespace ps
