// FP32 CG operator kernel of 3D meshes: one block per chunk and a completion
// block, star records staged by the TMA engine, shared-node inputs from a
// chunk-major halo.
//
// The same iteration step as k_cg2_chunks<3, float> (p = D^-1 r + beta p on
// the chunk's nodes, q = A p, the chunk's share of p.Ap), for meshes of many
// chunks:
//   * one thread moves the chunk's star records and incidence lists into
//     shared memory with bulk copies on one mbarrier (the whole chunk is in
//     flight at once, without registers); a thread takes its stars' records
//     from there and leaves their contributions in the same place;
//   * shared nodes' inputs come from a halo, contiguous per chunk; a thread has
//     all its nodes' loads in flight before any store;
//   * the chunk's p.Ap share is merged per warp and then across the warps by
//     one thread; the chunk block stores it and exits, and one extra block of
//     the grid sums the shares in chunk order and sets alpha (no fence,
//     counter or wait in the chunk blocks).
// The pass moves 24 bytes per tetrahedron (a closed star of six: 19 weights
// and 5 id words, 16 bytes; incidence lists 2.7; vectors and row sums) in 2.0
// warp instructions; it is bound by the latency of a block's phases (load,
// gather, stars, node sums) with 36 warps per SM: 4.4 TB/s on 112^3 and 160^3.
#pragma once
#include "cg2.cuh"

namespace ps {

// A chunk share not yet written: both words all ones (a NaN that no
// arithmetic produces; computed NaNs are 0x7fffffff).
__device__ __forceinline__ bool share_unset(float v) { return __float_as_uint(v) == 0xffffffffu; }

// The operator pass's completion, in one extra block launched after the
// chunk blocks: each chunk block stores its share of p.Ap over the share's
// "unset" pattern and exits (no fence, no counter, no wait).  This block
// polls the shares in chunk order until each is set (bounded), sums them in
// a fixed order and sets alpha = rz / p.Ap, and restores the unset pattern
// for the next launch.  The chunk blocks never wait for it, so they always
// complete; on timeout the error flag is set, alpha is left unchanged and
// the shares are reset all the same (and again, on the stream, at the start
// of the next CG run, in case a late chunk block wrote its share after).
template <int NT>
__device__ __noinline__ void share_reduce_alpha(const Cg2Args<float> &a, int n_chunks, int *err, int tid) {
    __shared__ float2 s_w[NT / 32];
    // eight 16-byte loads (two chunk shares each) in flight per thread:
    // thread t takes the chunk pairs j = t + NT (8 i + k), chunks 2j and
    // 2j + 1, into accumulator k, merged in k order (the share array holds
    // at least one entry past the last chunk, so the pair load stays inside)
    constexpr int kAcc = 8;
    DotF part[kAcc];
    float4 *pq4 = reinterpret_cast<float4 *>(a.pq);
    const int n_pairs = (n_chunks + 1) / 2;
    uint32_t polls = 0;
    bool ok = true;
    for (int j0 = tid; j0 < n_pairs; j0 += NT * kAcc) {
        float4 v[kAcc];
#pragma unroll
        for (int k = 0; k < kAcc; ++k) {
            const int j = j0 + NT * k;
            v[k] = j < n_pairs ? __ldcg(pq4 + j) : make_float4(0.f, 0.f, 0.f, 0.f);
        }
#pragma unroll
        for (int k = 0; k < kAcc; ++k) {
            const int j = j0 + NT * k;
            if (j >= n_pairs) continue;
            const bool two = 2 * j + 1 < n_chunks;
            // wait (bounded) for the shares of chunks 2j and 2j + 1
            while (ok && (share_unset(v[k].x) || share_unset(v[k].y) ||
                          (two && (share_unset(v[k].z) || share_unset(v[k].w))))) {
                if (++polls > kGridSpinLimit) {
                    ok = false;
                    break;
                }
                __nanosleep(64);
                v[k] = __ldcg(pq4 + j);
            }
            part[k].merge(v[k].x, v[k].y);
            if (two) part[k].merge(v[k].z, v[k].w);
        }
        if (!ok) break;
    }
    ok = __syncthreads_and(ok);   // every share read
    for (int j = tid; j < n_pairs; j += NT)
        __stcg(pq4 + j, make_float4(__uint_as_float(0xffffffffu), __uint_as_float(0xffffffffu),
                                    __uint_as_float(0xffffffffu), __uint_as_float(0xffffffffu)));
    if (!ok) {
        if (tid == 0) atomicOr(err, kErrGridTimeout);
        return;
    }
    DotF acc = part[0];
#pragma unroll
    for (int k = 1; k < kAcc; ++k) acc.merge(part[k].hi, part[k].lo);
    acc = warp_merge(acc);
    if ((tid & 31) == 0) s_w[tid >> 5] = make_float2(acc.hi, acc.lo);
    __syncthreads();
    if (tid == 0) {
        DotF t;
#pragma unroll
        for (int w = 0; w < NT / 32; ++w) t.merge(s_w[w].x, s_w[w].y);
        const double pq = (double)t.hi + (double)t.lo;
        CgState *st = a.st;
        st->pq = pq;
        if (!(pq > 0.0) || !isfinite(pq)) {
            st->status = kCgBreakdown;
            st->done = 1;
        } else {
            st->alpha = st->rz / pq;
        }
    }
}

// The chunk's share of p.Ap from its warps' sums, merged in order.
template <int NT>
__device__ __forceinline__ float2 chunk_share(const float2 *wdot) {
    DotF t;
#pragma unroll
    for (int w = 0; w < NT / 32; ++w) t.merge(wdot[w].x, wdot[w].y);
    return part_pack((double)t.hi + (double)t.lo);
}

// Threads per block and resident blocks per SM the kernel is compiled for (62
// KB of shared memory per 3,072-tet chunk: three blocks).  Measured per pass on
// Kuhn 64^3, 96^3, 112^3, 160^3: 384 threads 14.5, 30.2, 46.2, 127.3 us; 256
// threads 14.8, 31.2, 50.2, 134.2; 512 threads 16.0, 33.3, 50.5, 134.9; 128
// threads 15.4 (64^3), 66.8 (112^3).  Recomputing the element matrices from
// coordinates (packed FP32x2, 15 bytes and 3.3 warp instructions per
// tetrahedron) took 17.0, 35.5, 55.2, 139.0.
constexpr int kStarThreads = 384;

// Nodes of a chunk a thread gathers at once (the rest in further rounds).
template <int NT>
constexpr int kGatherNodes = 1024 / NT;

// K1 on the halo layout: one block of NT threads (128, 256 or 384) per chunk and
// one more block (the last) for the completion, MINB blocks per SM (the
// register budget of a thread).
template <int NT, int MINB>
__global__ void __launch_bounds__(NT, MINB) k_cg2_stars(MeshDev m, Cg2Args<float> a) {
    constexpr int kG = kGatherNodes<NT>;
    extern __shared__ __align__(128) unsigned char smem[];
    uint4 *s_rec = reinterpret_cast<uint4 *>(smem + m.sms.rec);
    const uint16_t *s_incp = reinterpret_cast<const uint16_t *>(smem + m.sms.incp);
    const uint16_t *s_inc = reinterpret_cast<const uint16_t *>(smem + m.sms.inc);
    float *s_val = reinterpret_cast<float *>(smem + m.sms.val);
    uint64_t *s_bar = reinterpret_cast<uint64_t *>(smem + m.sms.bar);
    __shared__ float s_beta;
    __shared__ int s_done;
    __shared__ float2 s_wdot[NT / 32];
    const int tid = threadIdx.x;
    if (blockIdx.x == (unsigned)m.n_chunks) {
        if (tid == 0) s_done = ld_flag(&a.st->done);
        __syncthreads();
        if (!s_done) share_reduce_alpha<NT>(a, m.n_chunks, m.err, tid);
        return;
    }
    const ChunkDesc cd = m.chunks[blockIdx.x];
    const int np = cd.n_patch, n_loc = cd.n_loc, n_int = cd.n_int;
    if (tid == 0) {
        const int done = a.st->done;
        s_done = done;
        s_beta = (float)a.st->beta;
        if (!done) {
            // (the buffers have seen no generic access: no proxy fence)
            mbar_init(s_bar, 1);
            fence_mbar_init();
            const uint32_t b_rec = (uint32_t)((np + kStarLanes - 1) / kStarLanes * m.srows) * (kStarLanes * 16u);
            const uint32_t b_incp = (uint32_t)((n_loc + 1 + kIncpPad - 1) / kIncpPad * kIncpPad) * 2u;
            const uint32_t b_inc = (uint32_t)((cd.n_inc + kIncPad - 1) / kIncPad * kIncPad) * 2u;
            mbar_arrive_expect_tx(s_bar, b_rec + b_incp + b_inc);
            if (m.stream)
                bulk_g2s_stream(s_rec, star_rec<3>(m, cd, 0), b_rec, s_bar);
            else
                bulk_g2s(s_rec, star_rec<3>(m, cd, 0), b_rec, s_bar);
            bulk_g2s(smem + m.sms.incp, m.incp + cd.incp_off, b_incp, s_bar);
            bulk_g2s(smem + m.sms.inc, m.inc_rec + cd.inc_off, b_inc, s_bar);
        }
    }
    // Interior nodes: D^-1, r, p contiguous from int_begin; shared nodes:
    // (D^-1 r, p) from the chunk's contiguous halo slots.  Every load of the
    // first round is issued before the block waits for beta.  No Dirichlet
    // mask is needed (D^-1 = 0 and r = 0 there and p starts at 0).
    float dv[kG], rv[kG], pv[kG];
    auto fetch = [&](int l0) {
#pragma unroll
        for (int k = 0; k < kG; ++k) {
            const int l = l0 + k * NT;
            dv[k] = rv[k] = pv[k] = 0.f;
            if (l < n_int) {
                const int g = cd.int_begin + l;
                dv[k] = __ldg(a.dinv + g);
                rv[k] = a.r[g];
                pv[k] = a.p[g];
            } else if (l < n_loc) {
                const float2 h = a.halo[cd.sh_off + (l - n_int)];
                dv[k] = 1.f;
                rv[k] = h.x;
                pv[k] = h.y;
            }
        }
    };
    fetch(tid);
    const float *mrow = chunk_mrow<float>(m, cd);
    float mr[kG];
#pragma unroll
    for (int k = 0; k < kG; ++k) mr[k] = tid + k * NT < n_loc ? __ldg(mrow + tid + k * NT) : 0.f;
    __syncthreads();
    if (s_done) return;
    const float beta = s_beta;
    for (int l0 = tid;;) {
#pragma unroll
        for (int k = 0; k < kG; ++k) {
            const int l = l0 + k * NT;
            if (l < n_loc) {
                // shared nodes: fma(beta, p, 1 * z) = fma(beta, p, z), the value K2 stores
                const float v = cg_dir(dv[k], rv[k], beta, pv[k]);
                s_val[l] = v;
                if (l < n_int) a.p[cd.int_begin + l] = v;
            }
        }
        l0 += kG * NT;
        if (l0 >= n_loc) break;
        fetch(l0);
    }
    {
        bool ok = mbar_wait_bounded(s_bar, 0);
        ok = __syncthreads_and(ok);   // also publishes val
        if (!ok) {
            if (tid == 0) atomicOr(m.err, kErrMbarTimeout);
            mbar_wait_bounded(s_bar, 0);
            return;
        }
    }
    for (int q = tid; q < np; q += NT) {
        uint4 *rec = s_rec + (q / kStarLanes) * (m.srows * kStarLanes) + q % kStarLanes;
        StarF<3> st;
        st.load_shared(rec);
        float out[12];
        star_eval<3>(st, s_val, out);
        float4 *o4 = reinterpret_cast<float4 *>(rec);
        o4[0] = make_float4(out[0], out[1], out[2], out[3]);
        o4[kStarLanes] = make_float4(out[4], out[5], out[6], out[7]);
        o4[2 * kStarLanes].x = out[8];
    }
    __syncthreads();
    DotF acc;
    const float *s_c = reinterpret_cast<const float *>(s_rec);
    auto emit = [&](int l, float mrl) {
        const float v = s_val[l];
        float s = fmaf(fabsf(mrl), v, list_sum(s_c, s_inc, s_incp[l], s_incp[l + 1]));
        acc.add_prod(v, s);                     // element-wise p^T A_e p over the chunk
        if (is_dirichlet(mrl)) s = 0.f;
        if (l < n_int)
            a.q[cd.int_begin + l] = s;
        else
            a.partial[__ldg(m.sh_dest + cd.sh_off + (l - n_int))] = s;
    };
#pragma unroll
    for (int k = 0; k < kG; ++k)
        if (tid + k * NT < n_loc) emit(tid + k * NT, mr[k]);
    for (int l = tid + kG * NT; l < n_loc; l += NT) emit(l, __ldg(mrow + l));
    acc = warp_merge(acc);
    if ((tid & 31) == 0) s_wdot[tid >> 5] = make_float2(acc.hi, acc.lo);
    __syncthreads();
    if (tid == 0) a.pq[blockIdx.x] = chunk_share<NT>(s_wdot);   // one 8-byte store over the unset pattern
}

// The halo of k_cg2_stars: every chunk-major shared slot j (node
// i = sh_ids[j]) gets (D^-1_i r_i, p_i) -- after each update kernel (the next
// operator pass reads it contiguously per chunk), at the start of a CG run
// and before ps_debug_cg_apply.  Pads (sh_ids = -1) are skipped.  Inside the
// iteration (reduce = 1) the first block instead sums the update kernel's
// block shares of rz and rr in block order and ends the iteration
// (cg2_update_tail), while the other blocks gather; a run that was already
// done before this iteration's update kernel does nothing.
static __global__ void __launch_bounds__(256) k_halo_gather(int64_t n_slots, const int32_t *__restrict__ sh_ids,
                                                            Cg2Args<float> a, int reduce) {
    if (reduce) {
        if (ld_flag(&a.st->done)) return;
        if (blockIdx.x == 0) {
            __shared__ double red[34];
            double rz, rr;
            part_sum2(a.z2, a.z2 + a.g3, a.g3, red, rz, rr);
            if (threadIdx.x == 0) cg2_update_tail(a.st, rz, rr);
            return;
        }
    }
    const int64_t b = reduce ? blockIdx.x - 1 : blockIdx.x, nb = reduce ? gridDim.x - 1 : gridDim.x;
    const float *__restrict__ r = a.r;
    const float *__restrict__ p = a.p;
    const float *__restrict__ dinv = a.dinv;
    for (int64_t j = b * blockDim.x + threadIdx.x; j < n_slots; j += nb * blockDim.x) {
        const int i = __ldg(sh_ids + j);
        if (i >= 0) a.halo[j] = make_float2(__fmul_rn(__ldg(dinv + i), r[i]), p[i]);
    }
}

}  // namespace ps
