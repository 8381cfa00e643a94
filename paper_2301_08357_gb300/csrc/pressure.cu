// libpressure: host side of the C ABI declared in include/pressure.h.
//
// Context and mesh objects, device memory accounting, coefficient upload, the
// matrix-free apply, and the single-mesh solvers (plain FP64 PCG; FP32 PCG
// inside FP64 defect correction).  CG iterations are captured once per mesh
// into CUDA graphs of `graph_iters` iterations; every kernel of an iteration
// first checks the device-side done flag, so a graph launched after
// convergence costs only its launch latency.
#include <cuda_runtime.h>

#include <chrono>
#include <cmath>
#include <cstdio>
#include <cstring>
#include <mutex>
#include <new>
#include <set>
#include <string>
#include <vector>

#include "../../include/pressure.h"
#include "internal.h"
#include "cg1.cuh"
#include "cg2.cuh"
#include "cg2s.cuh"

using namespace ps;

namespace ps {

const int kBlock = kChunkThreads;   // threads per block of every kernel
static const int kUpdateBlocksPerSm = 2;   // update-kernel grid when occupancy is unknown

// Star records beyond this size are read with evict-first priority by the
// operator kernel (half of the 129 MB L2: records, vectors and partial sums of
// a smaller mesh stay resident from one pass to the next).  Measured on Kuhn
// cubes, evict-first / plain: 64^3 (25 MB of records) 15.4 / 14.7 us per pass,
// 96^3 (85 MB) 31.3 / 38.8, 112^3 (135 MB) 50.4 / 54.9, 160^3 (393 MB) 134.9 /
// 135.7; the update kernel gains too (96^3: 11.1 -> 9.5 us).
static constexpr int64_t kStreamBytes = int64_t(64) << 20;

static int sm_count_of(int dev) {
    int v = 0;
    cudaDeviceGetAttribute(&v, cudaDevAttrMultiProcessorCount, dev);
    return v > 0 ? v : 1;
}

int grid_for(int64_t n, int dev_sms) {
    int64_t g = (n + kBlock - 1) / kBlock;
    int64_t cap = (int64_t)dev_sms * 4;
    if (g > cap) g = cap;
    if (g < 1) g = 1;
    return (int)g;
}

// ---- context-accounted device allocations
int dalloc(ps_ctx *ctx, void **p, size_t bytes, std::vector<DevAlloc> &owner) {
    *p = nullptr;
    if (bytes == 0) bytes = 16;
    bytes = (bytes + 255) / 256 * 256;
    if (ctx->budget && ctx->bytes + (int64_t)bytes > (int64_t)ctx->budget) return PS_ENOMEM;
    cudaError_t e = cudaMalloc(p, bytes);
    if (e != cudaSuccess) {
        cudaGetLastError();
        *p = nullptr;
        return PS_ENOMEM;
    }
    ctx->bytes += (int64_t)bytes;
    owner.push_back(DevAlloc{*p, bytes});
    return PS_OK;
}

void dfree_all(ps_ctx *ctx, std::vector<DevAlloc> &owner) {
    for (auto &a : owner) {
        cudaFree(a.p);
        ctx->bytes -= (int64_t)a.bytes;
    }
    owner.clear();
}

static uint32_t align128(uint64_t v) { return (uint32_t)((v + 127) / 128 * 128); }

// Geometry of element j of a star patch (vertices A, B, ring j, ring j+1 in
// 3D; A, ring j, ring j+1 in 2D; chunk-relative coordinates rel): the
// cofactor vectors c_a (grad lambda_a = c_a / det) and the slot words of
// kGeoWords.
static void element_geometry(int dim, const double *rel, const uint16_t *rec, int j, double *out) {
    auto P = [&](int l) { return rel + (size_t)l * dim; };
    if (dim == 3) {
        const double *A = P(rec[1]), *B = P(rec[2]), *R0 = P(rec[3 + j]), *R1 = P(rec[4 + j]);
        double e1[3], d0[3], d1[3], c[4][3];
        for (int k = 0; k < 3; ++k) {
            e1[k] = B[k] - A[k];
            d0[k] = R0[k] - A[k];
            d1[k] = R1[k] - A[k];
        }
        auto cross = [](const double *u, const double *v, double *w) {
            w[0] = u[1] * v[2] - u[2] * v[1];
            w[1] = u[2] * v[0] - u[0] * v[2];
            w[2] = u[0] * v[1] - u[1] * v[0];
        };
        cross(d0, d1, c[1]);   // B
        cross(d1, e1, c[2]);   // ring j
        cross(e1, d0, c[3]);   // ring j + 1
        for (int k = 0; k < 3; ++k) c[0][k] = -(c[1][k] + c[2][k] + c[3][k]);
        const double ad = std::fabs(e1[0] * c[1][0] + e1[1] * c[1][1] + e1[2] * c[1][2]);
        const double inv = 1.0 / (6.0 * ad);
        auto G = [&](int a, int b) { return (c[a][0] * c[b][0] + c[a][1] * c[b][1] + c[a][2] * c[b][2]) * inv; };
        out[0] = G(0, 1);
        out[1] = G(0, 2);
        out[2] = G(0, 3);
        out[3] = G(1, 2);
        out[4] = G(1, 3);
        out[5] = G(2, 3);
        out[6] = ad;
    } else {
        const double *A = P(rec[1]), *R0 = P(rec[3 + j]), *R1 = P(rec[4 + j]);
        const double d0[2] = {R0[0] - A[0], R0[1] - A[1]}, d1[2] = {R1[0] - A[0], R1[1] - A[1]};
        const double c[3][2] = {{-(d1[1] - d0[1]), -(-d1[0] + d0[0])}, {d1[1], -d1[0]}, {-d0[1], d0[0]}};
        const double ad = std::fabs(d0[0] * d1[1] - d0[1] * d1[0]);
        const double inv = 1.0 / (2.0 * ad);
        auto G = [&](int a, int b) { return (c[a][0] * c[b][0] + c[a][1] * c[b][1]) * inv; };
        out[0] = G(0, 1);
        out[1] = G(0, 2);
        out[2] = G(1, 2);
        out[3] = ad;
    }
}

SmemLayout make_layout(int esz, int max_loc, int max_patch, int max_inc) {
    SmemLayout L;
    const uint64_t ppad = (uint64_t)round_up(max_patch, kPatchPad);
    uint64_t off = 0;
    L.val = (uint32_t)off;     off += align128((uint64_t)max_loc * esz);
    L.aux = (uint32_t)off;     off += align128((uint64_t)max_loc * esz);
    L.incp = (uint32_t)off;    off += align128((uint64_t)round_up(max_loc + 1, kIncpPad) * 2);
    L.inc = (uint32_t)off;     off += align128((uint64_t)round_up(max_inc > 0 ? max_inc : 1, kIncPad) * 2);
    L.contrib = (uint32_t)off; off += align128(ppad * kPatchSlots * esz);
    L.red = (uint32_t)off;     off += 34 * 8;
    L.bar = (uint32_t)off;     off += 16;
    L.total = (uint32_t)off;
    return L;
}

// The largest chunk the interface takes: per local node 48 bytes, per patch
// 24 + 72 bytes, the incidence pointers and lists and 4 bytes per shared node
// within 227 KB (more than any pass stages; the limit does not move with the
// kernels' layouts).
static bool chunk_fits(const PrepMesh &pm) {
    const uint64_t ppad = (uint64_t)round_up(pm.max_patch, 4);
    uint64_t b = align128((uint64_t)pm.max_loc * 32) + 2 * align128((uint64_t)pm.max_loc * 8) + align128(ppad * 24) +
                 align128((uint64_t)round_up(pm.max_loc + 1, kIncpPad) * 2) +
                 align128((uint64_t)round_up(pm.max_inc > 0 ? pm.max_inc : 1, kIncPad) * 2) +
                 align128((uint64_t)round_up(pm.max_sh > 0 ? pm.max_sh : 1, kShPad) * 4) + align128(ppad * 72) +
                 34 * 8 + 16;
    return b <= 227 * 1024;
}

int cuda_status(cudaError_t e) {
    if (e == cudaSuccess) return PS_OK;
    return e == cudaErrorMemoryAllocation ? PS_ENOMEM : PS_ECUDA;
}

}  // namespace ps

#define CK(call)                                            \
    do {                                                    \
        cudaError_t _e = (call);                            \
        if (_e != cudaSuccess) {                            \
            ps_set_last_error(cudaGetErrorString(_e));      \
            return cuda_status(_e);                         \
        }                                                   \
    } while (0)

#define RC(call)                      \
    do {                              \
        int _r = (call);              \
        if (_r != PS_OK) return _r;   \
    } while (0)

static thread_local std::string g_last_error;
extern "C" void ps_set_last_error(const char *msg) { g_last_error = msg ? msg : ""; }
extern "C" const char *ps_last_error(void) { return g_last_error.c_str(); }

// ---------------------------------------------------------------- kernels setup
namespace ps {

// Largest dynamic shared memory next to the kernel's static shared memory.
template <typename F>
static cudaError_t set_max_dyn_smem(F *func) {
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

// Every kernel launched with a chunk's shared-memory layout (which can pass
// the 48 KB default for large chunks) gets the opt-in maximum.
static int set_smem_attrs() {
    CK(set_max_dyn_smem(k_chunks<2, float, kApply>));
    CK(set_max_dyn_smem(k_chunks<3, float, kApply>));
    CK(set_max_dyn_smem(k_chunks<2, double, kApply>));
    CK(set_max_dyn_smem(k_chunks<3, double, kApply>));
    CK(set_max_dyn_smem(k_chunks<2, double, kResid>));
    CK(set_max_dyn_smem(k_chunks<3, double, kResid>));
    CK(set_max_dyn_smem(k_star_build<2>));
    CK(set_max_dyn_smem(k_star_build<3>));
    CK(set_max_dyn_smem(k_cg1_chunks<2>));
    CK(set_max_dyn_smem(k_cg1_chunks<3>));
    CK(set_max_dyn_smem(k_cg2_chunks<2, float>));
    CK(set_max_dyn_smem(k_cg2_chunks<3, float>));
    CK(set_max_dyn_smem(k_cg2_chunks<2, double>));
    CK(set_max_dyn_smem(k_cg2_chunks<3, double>));
    CK(set_max_dyn_smem(k_cg2_stars<kStarThreads, 3>));
    CK(set_max_dyn_smem(k_cg2_stars<256, 3>));
    CK(set_max_dyn_smem(k_cg2_stars<128, 5>));
    RC(batched_set_attrs());
    return solo_set_attrs();
}

// Launch kernel 1 + kernel 2 of one operator pass (mode MODE, type T).
template <typename T, int MODE>
int launch_pass(ps_mesh *m, const VecArgs<T> &a, cudaStream_t s) {
    const SmemLayout &L = sizeof(T) == 4 ? m->dev.sm32 : m->dev.sm64;
    if (m->dev.dim == 2)
        k_chunks<2, T, MODE><<<m->dev.n_chunks, kBlock, L.total, s>>>(m->dev, a);
    else
        k_chunks<3, T, MODE><<<m->dev.n_chunks, kBlock, L.total, s>>>(m->dev, a);
    CK(cudaGetLastError());
    // Kernel 2's launch overlaps kernel 1 (apply 45^3 FP32: 12.3 -> 10.3 us per
    // call of a loop, 8.6 -> 7.9 in a graph).
    cudaLaunchConfig_t cfg;
    std::memset(&cfg, 0, sizeof(cfg));
    cfg.gridDim = dim3(m->grid2);
    cfg.blockDim = dim3(kBlock);
    cfg.stream = s;
    cudaLaunchAttribute attr[1];
    attr[0].id = cudaLaunchAttributeProgrammaticStreamSerialization;
    attr[0].val.programmaticStreamSerializationAllowed = 1;
    cfg.attrs = attr;
    cfg.numAttrs = 1;
    CK(cudaLaunchKernelEx(&cfg, k_shared<T, MODE>, m->dev, a, m->dev.n_chunks));
    m->launches += 2;
    return PS_OK;
}

// The chunk kernel reads x and writes interior rows of y through the caller's
// vertex of each local node, the second kernel the shared rows (and the
// vertices merged into them): two launches instead of four with a permuted
// copy of x before and of y after.  Measured per call, four / two launches:
// FP64 64 x 64 squares 20.5 / 12.3 us, FP32 45^3 20.5 / 12.3, FP64 112^3 238 / 221.
template <typename T>
int launch_apply(ps_mesh *m, const T *x, T *y, T *part, cudaStream_t s) {
    VecArgs<T> a;
    std::memset(&a, 0, sizeof(a));
    a.x = x;
    a.y = y;
    a.partial = part;
    a.loc_user = m->d_loc_user;
    a.old_of_new = m->d_old_of_new;
    a.slave_ptr = m->d_slave_ptr;
    a.slave = m->d_slave;
    return launch_pass<T, kApply>(m, a, s);
}
template int launch_apply<float>(ps_mesh *, const float *, float *, float *, cudaStream_t);
template int launch_apply<double>(ps_mesh *, const double *, double *, double *, cudaStream_t);
template int launch_pass<double, kResid>(ps_mesh *, const VecArgs<double> &, cudaStream_t);

}  // namespace ps

// ---------------------------------------------------------------- ABI: library / ctx
extern "C" const char *ps_version(void) { return "libpressure 0.1 (sm_103a)"; }

extern "C" const char *ps_status_str(int s) {
    switch (s) {
        case PS_OK: return "ok";
        case PS_PENDING: return "pending";
        case PS_EINVAL: return "invalid argument";
        case PS_ENOMEM: return "out of device memory / over HBM budget";
        case PS_ENOTCONV: return "not converged";
        case PS_EBREAKDOWN: return "CG breakdown";
        case PS_ETIMEOUT: return "device wait timed out";
        case PS_ECUDA: return "CUDA error";
        case PS_ESTATE: return "call out of order";
        case PS_ENOTFOUND: return "not found";
        default: return "unknown status";
    }
}

extern "C" int ps_ctx_create(ps_ctx **out, int device, size_t budget) {
    if (!out) return PS_EINVAL;
    *out = nullptr;
    int n = 0;
    CK(cudaGetDeviceCount(&n));
    if (device < 0 || device >= n) return PS_EINVAL;
    CK(cudaSetDevice(device));
    RC(set_smem_attrs());
    RC(noalloc_setup(device));
    ps_ctx *c = new (std::nothrow) ps_ctx();
    if (!c) return PS_ENOMEM;
    c->device = device;
    c->budget = budget;
    c->sms = sm_count_of(device);
    int *e = nullptr;
    if (cudaMalloc(&e, 64) != cudaSuccess) {
        delete c;
        return PS_ENOMEM;
    }
    cudaMemset(e, 0, 64);
    c->d_err = e;
    *out = c;
    return PS_OK;
}

extern "C" void ps_ctx_destroy(ps_ctx *c) {
    if (!c) return;
    cudaSetDevice(c->device);
    std::vector<ps_mesh *> ms(c->meshes.begin(), c->meshes.end());
    for (ps_mesh *m : ms) ps_mesh_free(m);
    cudaFree(c->d_err);
    if (c->d_bar) cudaFree(c->d_bar);
    delete c;
}

extern "C" int64_t ps_ctx_bytes_in_use(const ps_ctx *c) { return c ? (int64_t)c->bytes.load() : 0; }

// ---------------------------------------------------------------- ABI: mesh
template <typename V>
static int upload(ps_ctx *c, ps_mesh *m, V **dst, const void *src, size_t bytes) {
    void *p = nullptr;
    RC(dalloc(c, &p, bytes, m->allocs));
    if (src && bytes) CK(cudaMemcpy(p, src, bytes, cudaMemcpyHostToDevice));
    *dst = reinterpret_cast<V *>(p);
    return PS_OK;
}

static int mesh_upload_impl(ps_ctx *c, ps_mesh *m, const PrepMesh &pm) {
    MeshDev &d = m->dev;
    std::memset(&d, 0, sizeof(d));
    d.dim = pm.dim;
    d.n_chunks = pm.n_chunks;
    d.n_nodes = pm.n_dofs;             // internal vectors are per unknown
    d.n_int = pm.n_int;
    d.n_shared = pm.n_shared;
    d.n_pad = round_up(pm.n_dofs, 4);
    ChunkDesc *ch;
    RC(upload(c, m, &ch, pm.chunks.data(), pm.chunks.size() * sizeof(ChunkDesc)));
    d.chunks = ch;
    // star records: the ids in words 0..4, the weights when coefficients are set
    {
        int nv = pm.dim == 3 ? 6 : kStarVec<2>;
        for (int64_t q = 0; q < pm.patch_total; ++q)
            if (pm.dim == 3 && ((pm.sids[q * kStarIds + 4] >> 16) & 7u) == 7u) nv = kStarVec<3>;
        d.srows = nv;
        d.stream = (int64_t)pm.patch_total * nv * 16 > kStreamBytes;
        std::vector<uint32_t> rec((size_t)pm.patch_total * nv * 4, 0);
        for (int64_t q = 0; q < pm.patch_total; ++q)
            for (int k = 0; k < kStarIds; ++k)
                rec[(((size_t)(q / kStarLanes) * nv + k / 4) * kStarLanes + q % kStarLanes) * 4 + k % 4] =
                    pm.sids[q * kStarIds + k];
        uint4 *sr;
        RC(upload(c, m, &sr, rec.data(), rec.size() * 4));
        d.srec = sr;
    }
    uint16_t *u;
    RC(upload(c, m, &u, pm.incp.data(), pm.incp.size() * 2));
    d.incp = u;
    RC(upload(c, m, &u, pm.inc.data(), pm.inc.size() * 2));
    d.inc = u;
    int32_t *i32;
    RC(upload(c, m, &i32, pm.sh_ids.data(), pm.sh_ids.size() * 4));
    d.sh_ids = i32;
    RC(upload(c, m, &i32, pm.shr_ptr.data(), pm.shr_ptr.size() * 4));
    d.shr_ptr = i32;
    RC(upload(c, m, &i32, pm.sh_dest.data(), pm.sh_dest.size() * 4));
    d.sh_dest = i32;
    int4 *i4;
    RC(upload(c, m, &i4, pm.sh_info.data(), pm.sh_info.size() * 4));
    d.sh_info = i4;
    RC(upload(c, m, &m->d_loc_node, pm.loc_node.data(), pm.loc_node.size() * 4));
    {
        std::vector<int32_t> lu(pm.loc_total);
        for (int64_t k = 0; k < pm.loc_total; ++k) lu[k] = pm.old_of_new[pm.loc_node[k]];
        RC(upload(c, m, &m->d_loc_user, lu.data(), lu.size() * 4));
    }
    RC(upload(c, m, &m->d_elem_src, pm.elem_src.data(), pm.elem_src.size() * 4));
    RC(upload(c, m, &m->d_old_of_new, pm.old_of_new.data(), pm.old_of_new.size() * 4));
    RC(upload(c, m, &m->d_new_of_old, pm.new_of_old.data(), pm.new_of_old.size() * 4));
    if (!pm.slave.empty()) {
        RC(upload(c, m, &m->d_slave_ptr, pm.slave_ptr.data(), pm.slave_ptr.size() * 4));
        RC(upload(c, m, &m->d_slave, pm.slave.data(), pm.slave.size() * 4));
    }
    // Dirichlet flags, padded to n_pad with 1 so padding rows stay zero
    std::vector<uint8_t> dir(d.n_pad, 1);
    std::memcpy(dir.data(), pm.dirichlet_new.data(), pm.n_dofs);
    uint8_t *du;
    RC(upload(c, m, &du, dir.data(), dir.size()));
    d.dirichlet = du;
    // element geometry per patch slot (kGeoWords: stiffness weights G_ab =
    // c_a.c_b / (d! |det|) and |det|) from chunk-relative FP64 coordinates,
    // and the lumped weight of every local node over its chunk's elements
    {
        const int gw = pm.dim == 3 ? kGeoWords<3> : kGeoWords<2>;
        const double lf = pm.dim == 3 ? 1.0 / 24.0 : 1.0 / 6.0;
        std::vector<double> geo((size_t)pm.patch_total * kPatchMax * gw, 0.0), lump(pm.loc_total, 0.0);
        for (int ch = 0; ch < pm.n_chunks; ++ch) {
            const ChunkDesc &cd = pm.chunks[ch];
            const double *rel = &pm.loc_rel[(size_t)cd.node_off * pm.dim];
            double *gc = &geo[(size_t)cd.patch_off * kPatchMax * gw];
            for (int q = 0; q < cd.n_patch; ++q) {
                const uint16_t *rec = &pm.pids[(size_t)(cd.patch_off + q) * kPatchIds];
                for (int j = 0; j < rec[0]; ++j) {
                    double g[8];
                    element_geometry(pm.dim, rel, rec, j, g);
                    for (int k = 0; k < gw; ++k)
                        gc[((size_t)(q / kStarLanes * kPatchMax + j) * gw + k) * kStarLanes + q % kStarLanes] = g[k];
                    const double w = g[gw - 1] * lf;
                    lump[cd.node_off + rec[1]] += w;
                    if (pm.dim == 3) lump[cd.node_off + rec[2]] += w;
                    lump[cd.node_off + rec[3 + j]] += w;
                    lump[cd.node_off + rec[4 + j]] += w;
                }
            }
        }
        double *gp;
        RC(upload(c, m, &gp, geo.data(), geo.size() * 8));
        d.geo64 = gp;
        RC(upload(c, m, &m->d_lump, lump.data(), lump.size() * 8));
        std::vector<double> tot(d.n_pad, 0.0);
        for (int64_t k = 0; k < pm.loc_total; ++k) tot[pm.loc_node[k]] += lump[k];
        RC(upload(c, m, &m->d_lump_tot, tot.data(), tot.size() * 8));
    }
    float *f;
    double *g;
    double2 *sw;
    RC(upload(c, m, &sw, nullptr, pm.patch_total * (pm.dim == 3 ? kStarVec64<3> : kStarVec64<2>) * 16));
    CK(cudaMemset(sw, 0, pm.patch_total * (pm.dim == 3 ? kStarVec64<3> : kStarVec64<2>) * 16));   // (unused weights stay 0)
    d.sw64 = sw;
    RC(upload(c, m, &f, nullptr, pm.loc_total * 4));
    d.mrow32 = f;
    RC(upload(c, m, &g, nullptr, pm.loc_total * 8));
    d.mrow64 = g;
    RC(upload(c, m, &f, nullptr, d.n_pad * 4));
    d.mtot32 = f;
    RC(upload(c, m, &g, nullptr, d.n_pad * 8));
    d.mtot64 = g;
    RC(upload(c, m, &g, nullptr, pm.loc_total * 8));
    d.alpha64 = g;
    RC(upload(c, m, &g, nullptr, pm.patch_total * kPatchMax * 8));
    d.bdt2_64 = g;
    RC(upload(c, m, &f, nullptr, d.n_pad * 4));
    CK(cudaMemset(f, 0, d.n_pad * 4));
    d.dinv32 = f;
    RC(upload(c, m, &g, nullptr, d.n_pad * 8));
    CK(cudaMemset(g, 0, d.n_pad * 8));
    d.dinv64 = g;
    if (pm.dim == 3 && m->k1_variant != 1) {
        StarSmem &U = d.sms;
        uint32_t off = 0;
        auto take = [&](uint64_t bytes) {
            const uint32_t at = off;
            off = align128(off + bytes);
            return at;
        };
        const uint64_t groups = (pm.max_patch + kStarLanes - 1) / kStarLanes;
        U.rec = take(groups * d.srows * kStarLanes * 16);
        U.incp = take((uint64_t)round_up(pm.max_loc + 1, kIncpPad) * 2);
        U.inc = take((uint64_t)round_up(pm.max_inc > 0 ? pm.max_inc : 1, kIncPad) * 2);
        U.val = take((uint64_t)pm.max_loc * 4);
        U.bar = take(8);
        U.total = off;
        // incidence lists with the contributions' words in the records' place
        m->use_halo = U.total <= 200 * 1024 && groups * d.srows * kStarLanes * 4 < 65536;
        if (m->use_halo) {
            std::vector<uint16_t> inc(pm.inc.size());
            for (size_t k = 0; k < inc.size(); ++k) {
                const uint32_t q = pm.inc[k] / kPatchSlots, slot = pm.inc[k] % kPatchSlots;
                inc[k] = (uint16_t)(((q / kStarLanes * d.srows + slot / 4) * kStarLanes + q % kStarLanes) * 4 + slot % 4);
            }
            RC(upload(c, m, &u, inc.data(), inc.size() * 2));
            d.inc_rec = u;
        }
    }
    d.err = c->d_err;
    if (!chunk_fits(pm)) {
        ps_set_last_error("chunk too large for shared memory; lower chunk_elems");
        return PS_EINVAL;
    }
    d.sm32 = make_layout(4, pm.max_loc, pm.max_patch, pm.max_inc);
    d.sm64 = make_layout(8, pm.max_loc, pm.max_patch, pm.max_inc);
    m->grid2 = grid_for(pm.n_shared, c->sms);
    m->grid3 = grid_for(d.n_pad, c->sms);
    {
        // auto: one full wave of the update kernel (its resident blocks per
        // SM times the SMs); measured on 160^3: 33 us at 6 blocks/SM (one
        // wave) against 59 us at 2 and 43 us at 8 (a partial second wave)
        int64_t g = (d.n_pad / 4 + kBlock - 1) / kBlock;
        int bps = m->update_bps;
        if (bps <= 0) {
            int of = 0, od = 0;
            cudaError_t e1 = cudaOccupancyMaxActiveBlocksPerMultiprocessor(&of, k_cg2_update<float>, kBlock, 0);
            cudaError_t e2 = cudaOccupancyMaxActiveBlocksPerMultiprocessor(&od, k_cg2_update<double>, kBlock, 0);
            cudaGetLastError();
            bps = (e1 == cudaSuccess && e2 == cudaSuccess) ? std::min(of, od) : 0;
            if (bps <= 0) bps = kUpdateBlocksPerSm;
        }
        m->g3c = (int)std::max<int64_t>(1, std::min<int64_t>(g, (int64_t)bps * c->sms));
    }
    return PS_OK;
}

extern "C" int ps_mesh_upload(ps_ctx *c, int dim, int64_t n_nodes, const double *coords, int64_t n_elems,
                              const int32_t *conn, const uint8_t *dirichlet, const ps_mesh_opts *opts,
                              ps_mesh **out) {
    return ps_mesh_upload_periodic(c, dim, n_nodes, coords, n_elems, conn, dirichlet, nullptr, opts, out);
}

extern "C" int ps_mesh_upload_periodic(ps_ctx *c, int dim, int64_t n_nodes, const double *coords, int64_t n_elems,
                                       const int32_t *conn, const uint8_t *dirichlet, const int32_t *periodic,
                                       const ps_mesh_opts *opts, ps_mesh **out) {
    if (!c || !out || !coords || !conn) return PS_EINVAL;
    *out = nullptr;
    std::lock_guard<std::mutex> lk(c->mu);
    CK(cudaSetDevice(c->device));
    PrepOptions po;
    if (opts) {
        po.chunk_elems = opts->chunk_elems;
        po.chunk_nodes_max = opts->chunk_nodes_max;
    }
    po.periodic = periodic;
    // 3D meshes (operator kernel 2): the first wave's chunks
    // split in halves on one of every ~five resident blocks of an SM
    // (measured on 160^3 Kuhn with the kernel of the time: 141 -> 138 us per pass)
    const int sl = opts ? opts->split_lead : 0;
    if (sl < -1) return PS_EINVAL;
    if (sl > 0) po.split_lead = sl;
    else if (sl == 0 && dim == 3 && !(opts && opts->operator_kernel == 1)) po.split_lead = c->sms;
    ps_mesh *m = new (std::nothrow) ps_mesh();
    if (!m) return PS_ENOMEM;
    m->ctx = c;
    m->update_bps = opts ? opts->update_blocks_per_sm : 0;
    m->k1_variant = opts ? opts->operator_kernel : 0;
    const int ot = opts ? opts->operator_threads : 0;
    m->op_threads = ot;
    if (m->update_bps < 0 || m->update_bps > 64 || m->k1_variant < 0 || m->k1_variant > 2 ||
        (ot != 0 && ot != 128 && ot != 256)) {
        delete m;
        return PS_EINVAL;
    }
    std::string err = prepare_mesh(dim, n_nodes, coords, n_elems, conn, dirichlet, po, m->prep);
    if (!err.empty()) {
        ps_set_last_error(err.c_str());
        delete m;
        return PS_EINVAL;
    }
    int rc = mesh_upload_impl(c, m, m->prep);
    if (rc == PS_OK) rc = solo_upload(m);
    if (rc != PS_OK) {
        solo_release(m);
        dfree_all(c, m->allocs);
        delete m;
        return rc;
    }
    // coordinates in the caller's numbering (the projection stage's element
    // passes); host copies that are no longer needed are dropped
    m->coords_host.assign(coords, coords + n_nodes * dim);
    m->prep.loc_rel.clear();
    m->prep.loc_rel.shrink_to_fit();
    c->meshes.insert(m);
    *out = m;
    return PS_OK;
}

static void free_graphs(ps_mesh *m) {
    for (auto &g : m->ws.graphs)
        if (g.exec) cudaGraphExecDestroy(g.exec);
    m->ws.graphs.clear();
}

static void free_workspace(ps_mesh *m) {
    Workspace &w = m->ws;
    free_graphs(m);
    if (w.cap_stream) cudaStreamDestroy(w.cap_stream);
    w.cap_stream = nullptr;
    if (w.h_st) cudaFreeHost(w.h_st);
    w.h_st = nullptr;
    dfree_all(m->ctx, w.allocs);
    w.ready = false;
}

extern "C" void ps_mesh_free(ps_mesh *m) {
    if (!m) return;
    ps_ctx *c = m->ctx;
    std::lock_guard<std::mutex> lk(c->mu);
    cudaSetDevice(c->device);
    cudaDeviceSynchronize();
    free_workspace(m);
    batched_release_mesh(m);
    projection_release(m);
    solo_release(m);
    dfree_all(c, m->allocs);
    c->meshes.erase(m);
    delete m;
}

extern "C" int ps_mesh_get_stats(const ps_mesh *m, ps_mesh_stats *o) {
    if (!m || !o) return PS_EINVAL;
    std::memset(o, 0, sizeof(*o));
    const PrepMesh &p = m->prep;
    o->n_nodes = p.n_nodes;
    o->n_elems = p.n_elems;
    o->n_free = p.n_free;
    o->dim = p.dim;
    o->n_chunks = p.n_chunks;
    o->n_shared = p.n_shared;
    o->chunk_node_refs = p.loc_total;
    int64_t b = 0;
    for (auto &a : m->allocs) b += (int64_t)a.bytes;
    for (auto &a : m->ws.allocs) b += (int64_t)a.bytes;
    o->device_bytes = b;
    o->max_chunk_elems = p.max_elem;
    o->max_chunk_nodes = p.max_loc;
    o->solve_bytes = batch_ws_bytes(m);
    o->operator_kernel = m->use_halo ? 2 : 1;
    return PS_OK;
}

// ---------------------------------------------------------------- ABI: coefficients
// Star weights, row sums and Jacobi diagonal (d.dinv32, d.dinv64) from the
// mesh's alpha and beta (null: the beta*dt^2 stored last), on stream s.
// partial: scratch of two values per shared slot.
static void launch_star_build(ps_mesh *m, const MeshDev &d, const double *beta, double dt2, double *partial,
                              cudaStream_t s) {
    const int64_t n_part = m->prep.sh_total;
    if (d.dim == 2)
        k_star_build<2><<<d.n_chunks, kBlock, d.sm64.total, s>>>(d, m->d_elem_src, beta, dt2, partial, n_part);
    else
        k_star_build<3><<<d.n_chunks, kBlock, d.sm64.total, s>>>(d, m->d_elem_src, beta, dt2, partial, n_part);
    VecArgs<double> a;
    std::memset(&a, 0, sizeof(a));
    a.partial = partial;
    k_shared<double, kDiag><<<m->grid2, kBlock, 0, s>>>(d, a, (int)n_part);
}

static int coeff_upload(ps_mesh *m, const double *alpha, const double *beta, double dt2) {
    ps_ctx *c = m->ctx;
    const PrepMesh &p = m->prep;
    MeshDev &d = m->dev;
    std::vector<DevAlloc> tmp;
    void *dbeta = nullptr;
    int rc = dalloc(c, &dbeta, p.n_elems * 8, tmp);
    if (rc != PS_OK) return rc;
    cudaError_t e = cudaMemcpy(dbeta, beta, p.n_elems * 8, cudaMemcpyHostToDevice);
    if (e == cudaSuccess && alpha) {
        std::vector<double> an(p.n_dofs);   // the master vertex's alpha per unknown
        for (int64_t g = 0; g < p.n_dofs; ++g) an[g] = alpha[p.old_of_new[g]];
        void *dal = nullptr;
        rc = dalloc(c, &dal, p.n_dofs * 8, tmp);
        if (rc != PS_OK) {
            dfree_all(c, tmp);
            return rc;
        }
        e = cudaMemcpy(dal, an.data(), p.n_dofs * 8, cudaMemcpyHostToDevice);
        if (e == cudaSuccess) {
            k_set_alpha<<<grid_for(p.loc_total, c->sms), kBlock>>>(d, p.loc_total, m->d_loc_node, (const double *)dal);
            e = cudaGetLastError();
        }
    }
    if (e == cudaSuccess) {
        // star weights, row sums and the Jacobi diagonal (FP64 arithmetic, both precisions stored)
        void *part = nullptr;
        rc = dalloc(c, &part, (p.sh_total > 0 ? p.sh_total : 1) * 16, tmp);
        if (rc != PS_OK) {
            dfree_all(c, tmp);
            return rc;
        }
        launch_star_build(m, d, (const double *)dbeta, dt2, (double *)part, nullptr);
        e = cudaGetLastError();
        if (e == cudaSuccess) e = cudaDeviceSynchronize();
    }
    dfree_all(c, tmp);
    if (e != cudaSuccess) {
        ps_set_last_error(cudaGetErrorString(e));
        return cuda_status(e);
    }
    int herr = 0;
    CK(cudaMemcpy(&herr, c->d_err, sizeof(int), cudaMemcpyDeviceToHost));
    if (herr) {
        cudaMemset(c->d_err, 0, sizeof(int));
        return PS_ETIMEOUT;
    }
    m->dt2 = dt2;
    m->coeff_ok = true;
    return PS_OK;
}

extern "C" int ps_coeff_set(ps_mesh *m, const double *alpha, const double *beta, double dt2) {
    if (!m || !alpha || !beta) return PS_EINVAL;
    if (!(dt2 > 0.0) || !std::isfinite(dt2)) return PS_EINVAL;
    const PrepMesh &p = m->prep;
    for (int64_t i = 0; i < p.n_nodes; ++i)
        if (!(alpha[i] >= 0.0) || !std::isfinite(alpha[i])) return PS_EINVAL;
    for (int64_t e = 0; e < p.n_elems; ++e)
        if (!(beta[e] > 0.0) || !std::isfinite(beta[e])) return PS_EINVAL;
    std::lock_guard<std::mutex> lk(m->ctx->mu);
    CK(cudaSetDevice(m->ctx->device));
    int rc = coeff_upload(m, alpha, beta, dt2);
    if (rc == PS_OK) {
        m->alpha_set = true;
        m->alpha_newton = false;
        m->alpha_host.assign(alpha, alpha + p.n_nodes);
        m->alpha_version += 1;
    }
    return rc;
}

extern "C" int ps_coeff_set_beta(ps_mesh *m, const double *beta) {
    if (!m || !beta) return PS_EINVAL;
    if (!m->alpha_set) return PS_ESTATE;
    const PrepMesh &p = m->prep;
    for (int64_t e = 0; e < p.n_elems; ++e)
        if (!(beta[e] > 0.0) || !std::isfinite(beta[e])) return PS_EINVAL;
    std::lock_guard<std::mutex> lk(m->ctx->mu);
    CK(cudaSetDevice(m->ctx->device));
    return coeff_upload(m, nullptr, beta, m->dt2);
}

// ---------------------------------------------------------------- workspace
namespace ps {

// Star weights, row sums and Jacobi diagonal from the mesh's current alpha,
// beta (null: the stored beta*dt^2) and mass form, on stream s (FP64 element
// arithmetic, both precisions stored).  The caller holds the context mutex
// and the workspace exists.
static int star_update_device(ps_mesh *m, const double *beta, double dt2, cudaStream_t s) {
    const MeshDev &d = m->dev;
    launch_star_build(m, d, beta, dt2, m->ws.part64, s);
    CK(cudaGetLastError());
    return PS_OK;
}

// The same while the preconditioner keeps its diagonal: the current one goes
// into scratch (two free workspace vectors).
static int star_update_keep_diag(ps_mesh *m, cudaStream_t s) {
    MeshDev d2 = m->dev;
    d2.dinv64 = m->ws.q64;
    d2.dinv32 = m->ws.q32;
    launch_star_build(m, d2, nullptr, 0.0, m->ws.part64, s);
    CK(cudaGetLastError());
    return PS_OK;
}

// beta (caller's element order, device) -> beta*dt^2 per patch slot, star
// weights and the Jacobi diagonal, on stream s without allocating or
// synchronising (the projection stage updates the operator between Picard
// iterations).  diag = false: only the beta*dt^2 are stored; the caller's
// alpha update that follows (diag = true) forms the rest.  The caller holds
// the context mutex.
int beta_update_device(ps_mesh *m, const double *beta_dev, double dt2, cudaStream_t s, bool diag) {
    RC(ensure_workspace(m));
    const PrepMesh &p = m->prep;
    MeshDev &d = m->dev;
    if (!diag) {
        const int64_t nslots = p.patch_total * kPatchMax;
        k_set_beta<<<grid_for(nslots, m->ctx->sms), kBlock, 0, s>>>(nslots, m->d_elem_src, beta_dev, dt2,
                                                                     const_cast<double *>(d.bdt2_64));
    }
    CK(cudaGetLastError());
    m->dt2 = dt2;
    return diag ? star_update_device(m, beta_dev, dt2, s) : PS_OK;
}

// Nodal alpha (caller's numbering, device; each unknown takes its master
// vertex's value), then the star weights and (diag) the Jacobi diagonal; on
// stream s without allocating or synchronising.  Without diag a lumped
// operator only needs its row sums scaled.  The caller holds the context
// mutex.
int alpha_update_device(ps_mesh *m, const double *alpha_dev, cudaStream_t s, bool diag) {
    RC(ensure_workspace(m));
    const PrepMesh &p = m->prep;
    MeshDev &d = m->dev;
    k_set_alpha_user<<<grid_for(p.loc_total, m->ctx->sms), kBlock, 0, s>>>(
        d, p.loc_total, m->d_loc_node, m->d_old_of_new, alpha_dev, d.lumped && !diag ? m->d_lump : nullptr,
        m->d_lump_tot);
    CK(cudaGetLastError());
    if (diag) return star_update_device(m, nullptr, 0.0, s);
    return d.lumped ? PS_OK : star_update_keep_diag(m, s);
}

int ensure_workspace(ps_mesh *m) {
    Workspace &w = m->ws;
    if (w.ready) return PS_OK;
    ps_ctx *c = m->ctx;
    const int64_t np = m->dev.n_pad;
    const int64_t sh = m->prep.sh_total > 0 ? m->prep.sh_total : 1;
    void *p;
    auto A = [&](void **dst, size_t bytes) -> int {
        int r = dalloc(c, dst, bytes, w.allocs);
        if (r == PS_OK) cudaMemset(*dst, 0, bytes);
        return r;
    };
    int rc = PS_OK;
#define WA(field, T, n)                                   \
    if (rc == PS_OK) {                                    \
        rc = A(&p, (size_t)(n) * sizeof(T));              \
        w.field = (T *)p;                                 \
    }
    WA(x64, double, np);
    WA(b64, double, np);
    WA(r64, double, np);
    WA(p64, double, np);
    WA(q64, double, np);
    WA(x32, float, np);
    WA(r32, float, np);
    WA(p32, float, np);
    WA(q32, float, np);
    WA(part32, float, sh);
    WA(part64, double, 2 * sh);
    WA(dot1, double, m->dev.n_chunks + m->grid2 + 8);
    WA(dot2, double, 2 * m->grid3 + 8);
    WA(st, CgState, 1);
    WA(pq2, double, m->dev.n_chunks + 8);
    WA(z3, double, 6 * m->g3c + 8);
    WA(x32b, float, np);
    WA(r32b, float, np);
    WA(p32b, float, np);
    WA(q32b, float, np);
    WA(s32a, float, np);
    WA(s32b, float, np);
    WA(part32b, float, sh);
    WA(dots1, double, 3 * m->dev.n_chunks + 8);
    if (m->use_halo) WA(halo32, float2, sh);
    if (m->use_halo) WA(pqu, float2, m->dev.n_chunks + 8);
#undef WA
    if (rc != PS_OK) {
        dfree_all(c, w.allocs);
        return rc;
    }
    if (w.pqu) CK(cudaMemset(w.pqu, 0xff, ((size_t)m->dev.n_chunks + 8) * sizeof(float2)));
    CK(cudaHostAlloc((void **)&w.h_st, sizeof(CgState), cudaHostAllocDefault));
    CK(cudaStreamCreateWithFlags(&w.cap_stream, cudaStreamNonBlocking));
    w.ready = true;
    return PS_OK;
}

template <typename T>
static Cg2Args<T> cg2_args(ps_mesh *m) {
    Workspace &w = m->ws;
    Cg2Args<T> a;
    std::memset(&a, 0, sizeof(a));
    if (sizeof(T) == 4) {
        a.x = (T *)w.x32;
        a.r = (T *)w.r32;
        a.p = (T *)w.p32;
        a.q = (T *)w.q32;
        a.dinv = (const T *)m->dev.dinv32;
        a.partial = (T *)w.part32;
    } else {
        a.x = (T *)w.x64;
        a.r = (T *)w.r64;
        a.p = (T *)w.p64;
        a.q = (T *)w.q64;
        a.dinv = (const T *)m->dev.dinv64;
        a.partial = (T *)w.part64;
    }
    a.pq = (typename PartOf<T>::type *)w.pq2;
    if (sizeof(T) == 4 && m->use_halo) a.pq = (typename PartOf<T>::type *)w.pqu;
    a.z2 = (typename PartOf<T>::type *)w.z3;
    a.g3 = m->g3c;
    a.st = w.st;
    a.halo = (sizeof(T) == 4 && m->use_halo) ? w.halo32 : nullptr;
    return a;
}

// k_cg2_stars' chunk shares of p.Ap back to their "unset"
// pattern, on stream s: at the start of every CG run and before a diagnostic
// launch, so that no share written after an interrupted launch can be taken
// for a later one.
static cudaError_t reset_shares(ps_mesh *m, cudaStream_t s) {
    if (!m->ws.pqu) return cudaSuccess;
    return cudaMemsetAsync(m->ws.pqu, 0xff, ((size_t)m->dev.n_chunks + 8) * sizeof(float2), s);
}

// FP32 operator kernel of the two-kernel iteration (block sizes: see
// kStarThreads).
static void launch_k1_f32(ps_mesh *m, const Cg2Args<float> &a, cudaStream_t s) {
    const MeshDev &d = m->dev;
    if (m->use_halo) {
        const int g = d.n_chunks + 1;   // the chunks and the completion block
        if (m->op_threads == 128)
            k_cg2_stars<128, 5><<<g, 128, d.sms.total, s>>>(d, a);
        else if (m->op_threads == 256)
            k_cg2_stars<256, 3><<<g, 256, d.sms.total, s>>>(d, a);
        else
            k_cg2_stars<kStarThreads, 3><<<g, kStarThreads, d.sms.total, s>>>(d, a);
    } else {
        if (d.dim == 2) k_cg2_chunks<2, float><<<d.n_chunks, kBlock, d.sm32.total, s>>>(d, a);
        else k_cg2_chunks<3, float><<<d.n_chunks, kBlock, d.sm32.total, s>>>(d, a);
    }
}

static CG1Vec cg1_vec(ps_mesh *m) {
    Workspace &w = m->ws;
    CG1Vec v;
    v.x[0] = w.x32;
    v.x[1] = w.x32b;
    v.r[0] = w.r32;
    v.r[1] = w.r32b;
    v.s[0] = w.s32a;
    v.s[1] = w.s32b;
    v.p[0] = w.p32;
    v.p[1] = w.p32b;
    v.w[0] = w.q32;
    v.w[1] = w.q32b;
    v.part[0] = w.part32;
    v.part[1] = w.part32b;
    v.dinv = m->dev.dinv32;
    v.dots = reinterpret_cast<float2 *>(w.dots1);
    return v;
}

static void launch_cg1(ps_mesh *m, const CG1Vec &v, cudaStream_t s) {
    if (m->dev.dim == 2)
        k_cg1_chunks<2><<<m->dev.n_chunks, kBlock, m->dev.sm32.total, s>>>(m->dev, v, m->ws.st);
    else
        k_cg1_chunks<3><<<m->dev.n_chunks, kBlock, m->dev.sm32.total, s>>>(m->dev, v, m->ws.st);
}

// Enqueue `iters` CG iterations (no host sync) of precision T; FP32 with
// `fused` runs one fused pass per iteration.
template <typename T>
static int enqueue_cg_iters(ps_mesh *m, int iters, bool fused, cudaStream_t s) {
    if (sizeof(T) == 4 && fused) {
        const CG1Vec v = cg1_vec(m);
        for (int k = 0; k < iters; ++k) {
            launch_cg1(m, v, s);
            m->launches += 1;
            CK(cudaGetLastError());
        }
        return PS_OK;
    }
    const Cg2Args<T> a = cg2_args<T>(m);
    const SmemLayout &L = sizeof(T) == 4 ? m->dev.sm32 : m->dev.sm64;
    for (int k = 0; k < iters; ++k) {
        if (sizeof(T) == 4)
            launch_k1_f32(m, reinterpret_cast<const Cg2Args<float> &>(a), s);
        else if (m->dev.dim == 2)
            k_cg2_chunks<2, T><<<m->dev.n_chunks, kBlock, L.total, s>>>(m->dev, a);
        else
            k_cg2_chunks<3, T><<<m->dev.n_chunks, kBlock, L.total, s>>>(m->dev, a);
        k_cg2_update<T><<<m->g3c, kBlock, 0, s>>>(m->dev, a);
        m->launches += 2;
        if (sizeof(T) == 4 && a.halo) {
            const Cg2Args<float> &af = reinterpret_cast<const Cg2Args<float> &>(a);
            k_halo_gather<<<grid_for(m->prep.sh_total, m->ctx->sms) + 1, kBlock, 0, s>>>(m->prep.sh_total,
                                                                                        m->dev.sh_ids, af, 1);
            m->launches += 1;
        }
        CK(cudaGetLastError());
    }
    return PS_OK;
}

// Run CG iterations until the device state says done: graph batches of at
// most `gi` iterations (lengths below), each followed by a copy of the state
// to pinned host memory; gi <= 0 launches kernels directly.
template <typename T>
static int run_cg_until_done(ps_mesh *m, int gi, bool jac, bool fused, cudaStream_t s) {
    Workspace &w = m->ws;
    fused = fused && sizeof(T) == 4;
    const int kind = (sizeof(T) == 4 ? 0 : 1) + (jac ? 0 : 2) + (fused ? 4 : 0);
    const int per_iter = fused ? 1 : (sizeof(T) == 4 && m->use_halo ? 3 : 2);
    if (gi <= 0) {
        const int batch = 15;
        for (;;) {
            RC(enqueue_cg_iters<T>(m, batch, fused, s));
            CK(cudaMemcpyAsync(w.h_st, w.st, sizeof(CgState), cudaMemcpyDeviceToHost, s));
            CK(cudaStreamSynchronize(s));
            if (w.h_st->done) return PS_OK;
        }
    }
    // Graph lengths follow the iteration count of this kind's previous run on
    // the mesh (successive CG runs of one mesh need similar counts): the
    // first launches cover that count in graphs of at most gi iterations,
    // rounded up to 4; past it, graphs of 4, 8, 16, ... iterations.  A
    // converged state makes the remaining iterations of a graph return at
    // once, so this only trims those idle launches.  Lengths are multiples
    // of 4 up to gi: a handful of captured graphs per kind.
    auto graph_of = [&](int len, GraphRec **out) -> int {
        for (auto &r : w.graphs)
            if (r.kind == kind && r.iters == len) {
                *out = &r;
                return PS_OK;
            }
        cudaGraph_t graph;
        CK(cudaStreamBeginCapture(w.cap_stream, cudaStreamCaptureModeThreadLocal));
        const int64_t saved_launches = m->launches;
        int rc = enqueue_cg_iters<T>(m, len, fused, w.cap_stream);
        m->launches = saved_launches;
        cudaError_t e2 = cudaMemcpyAsync(w.h_st, w.st, sizeof(CgState), cudaMemcpyDeviceToHost, w.cap_stream);
        cudaError_t e = cudaStreamEndCapture(w.cap_stream, &graph);
        if (rc != PS_OK) return rc;
        CK(e2);
        CK(e);
        cudaGraphExec_t ex;
        e = cudaGraphInstantiate(&ex, graph, 0);
        cudaGraphDestroy(graph);
        CK(e);
        w.graphs.push_back(GraphRec{kind, len, ex});
        *out = &w.graphs.back();
        return PS_OK;
    };
    const int64_t hint = w.last_iters[kind];
    int64_t ran = 0;
    int extra = 0;
    for (;;) {
        int len = gi;
        if (hint > 0) {
            const int64_t rem = hint - ran;
            len = rem > 0 ? (int)std::min<int64_t>(gi, (rem + 3) / 4 * 4) : std::min(gi, 4 << std::min(extra++, 8));
            len = std::max(1, std::min(len, gi));
        }
        GraphRec *g = nullptr;
        RC(graph_of(len, &g));
        CK(cudaGraphLaunch(g->exec, s));
        m->launches += per_iter * (int64_t)len;
        CK(cudaStreamSynchronize(s));
        ran += len;
        if (w.h_st->done) {
            w.last_iters[kind] = w.h_st->iters;
            return PS_OK;
        }
    }
}

static int read_state(ps_mesh *m, cudaStream_t s, CgState *out) {
    CK(cudaMemcpyAsync(m->ws.h_st, m->ws.st, sizeof(CgState), cudaMemcpyDeviceToHost, s));
    CK(cudaStreamSynchronize(s));
    *out = *m->ws.h_st;
    return PS_OK;
}

// FP64 true residual r64 = b64 - A x64; returns ||r||^2 (free nodes).
static int true_residual(ps_mesh *m, cudaStream_t s, double *rr) {
    Workspace &w = m->ws;
    VecArgs<double> a;
    std::memset(&a, 0, sizeof(a));
    a.x = w.x64;
    a.y = w.r64;
    a.b = w.b64;
    a.partial = w.part64;
    a.dotbuf = w.dot1;
    a.st = w.st;
    RC((launch_pass<double, kResid>(m, a, s)));
    CgState h;
    RC(read_state(m, s, &h));
    *rr = h.rr;
    return PS_OK;
}

static int check_dev_err(ps_ctx *c) {
    int herr = 0;
    CK(cudaMemcpy(&herr, c->d_err, sizeof(int), cudaMemcpyDeviceToHost));
    if (herr) {
        cudaMemset(c->d_err, 0, sizeof(int));
        return PS_ETIMEOUT;
    }
    return PS_OK;
}

// PS_ENGINE_AUTO where a mixed solve cannot run on chip (regular meshes of this
// size only when the context has no room for its workspace): the fused pass up
// to here, the two-kernel iteration above.  Per iteration, fused / two-kernel, in
// us: 2D 4,225 nodes 11.8 / 16.3, 91,204 15.7 / 17.2, 251,001 17.0 / 18.4,
// 491,401 26.8 / 26.1; 3D 35,937 20.6 / 18.4, 97,336 16.5 / 18.0, 148,877 24.4 /
// 20.6, 274,625 33.9 / 25.4.
static constexpr int64_t kFusedMaxNodes = 200000;

}  // namespace ps

// Relative reduction asked of an inner FP32 solve of the mixed solver: the
// configured one, or, when the outer residual is already close to the
// target, only what is still needed times 0.1 (at most 0.5).  ||r||^2 = rr,
// ||b||^2 = bb.
double ps::inner_reduction(double itol, double tol, double bb, double rr) {
    if (!(rr > 0.0)) return itol;
    const double need = 0.1 * tol * std::sqrt(bb > 0.0 ? bb : 1.0) / std::sqrt(rr);
    return need > itol ? std::min(need, 0.5) : itol;
}

namespace ps {

int solve_internal(ps_mesh *m, const ps_solve_opts &o, ps_solve_info *info, cudaStream_t s) {
    Workspace &w = m->ws;
    const int64_t np = m->dev.n_pad;
    const int g3 = m->grid3;
    // ||b||^2 through the residual pass with x = 0 would cost an apply; use a
    // start kernel on b instead (rz unused).
    k_cg_start<double><<<g3, kBlock, 0, s>>>(np, w.b64, 1.0, w.r64, nullptr, w.p64, m->dev.dinv64, w.st, w.dot2, 0.0,
                                             0, 0);
    CK(cudaGetLastError());
    m->launches += 1;
    CgState h;
    RC(read_state(m, s, &h));
    const double bb = h.rr0;
    info->bnorm = std::sqrt(bb);
    info->n_free = m->prep.n_free;
    const double tol = o.tol > 0 ? o.tol : 1e-10;
    const double stop_abs2 = tol * tol * (bb > 0 ? bb : 1.0);
    const int64_t max_it = o.max_iters > 0 ? o.max_iters : 100000;
    int64_t used = 0, outer = 0;
    double rr = 0;
    int status = PS_ENOTCONV;
    const bool jac = o.precond != PS_PRECOND_NONE;
    const float *dinv32 = m->dev.dinv32;
    const double *dinv64 = m->dev.dinv64;
    if (!jac) {
        // unpreconditioned: D^-1 = 1 on free nodes (kept in a workspace vector)
        if (!w.ones_ready) {
            RC(dalloc(m->ctx, (void **)&w.one32, np * 4, w.allocs));
            RC(dalloc(m->ctx, (void **)&w.one64, np * 8, w.allocs));
            std::vector<float> f(np);
            std::vector<double> d(np);
            std::vector<uint8_t> dir(np, 1);
            for (int64_t i = 0; i < m->prep.n_dofs; ++i) dir[i] = m->prep.dirichlet_new[i];
            for (int64_t i = 0; i < np; ++i) {
                f[i] = dir[i] ? 0.f : 1.f;
                d[i] = dir[i] ? 0.0 : 1.0;
            }
            CK(cudaMemcpy(w.one32, f.data(), np * 4, cudaMemcpyHostToDevice));
            CK(cudaMemcpy(w.one64, d.data(), np * 8, cudaMemcpyHostToDevice));
            w.ones_ready = true;
        }
        dinv32 = w.one32;
        dinv64 = w.one64;
    }
    MeshDev saved = m->dev;
    m->dev.dinv32 = dinv32;
    m->dev.dinv64 = dinv64;
    const int gi = o.graph_iters == 0 ? 32 : o.graph_iters;
    const uint32_t spin = o.grid_spin_limit > 0 ? (uint32_t)o.grid_spin_limit : kGridSpinLimit;
    int rc = PS_OK;
    if (o.mode == PS_MODE_FP64) {
        const int max_restarts = o.max_outer > 0 ? o.max_outer : 40;
        const bool solo = o.engine == PS_ENGINE_AUTO && m->solo && m->solo->fp64 && solo_ready(m);
        for (;;) {
            rc = true_residual(m, s, &rr);
            if (rc != PS_OK) break;
            ++outer;
            if (rr <= stop_abs2) { status = PS_OK; break; }
            if (used >= max_it || outer > max_restarts) { status = PS_ENOTCONV; break; }
            if (solo) {
                // r scaled by a power of two to a norm near 1 (every number of the
                // run is the same but for its exponent): the quotients are formed
                // from products of two dot products, which would leave the range of
                // a double for right-hand sides of 1e80 or 1e-80
                int e = 0;
                if (std::isfinite(rr)) std::frexp(std::sqrt(rr), &e);
                rc = solo_run<double>(m, std::ldexp(1.0, -e), std::ldexp(stop_abs2, -2 * e), max_it - used, true, spin, s);
                if (rc != PS_OK) break;
            } else {
                Cg2Args<double> a = cg2_args<double>(m);
                k_cg2_start<double><<<m->g3c, kBlock, 0, s>>>(m->dev, a, nullptr, 1.0, nullptr, stop_abs2, 0,
                                                              max_it - used);
                m->launches += 1;
            }
            if ((rc = cuda_status(cudaGetLastError())) != PS_OK) break;
            if (!solo && (rc = run_cg_until_done<double>(m, gi, jac, false, s)) != PS_OK) break;
            RC(read_state(m, s, &h));
            if (solo) solo_end(*m->solo, h.done != 0, h.iters);
            if (solo && !h.done) { rc = PS_ETIMEOUT; break; }
            used += h.iters;
            if (h.status == kCgBreakdown) { status = PS_EBREAKDOWN; rc = PS_OK; break; }
        }
    } else {
        const double itol = o.inner_tol > 0 ? o.inner_tol : 1e-4;
        const int max_outer = o.max_outer > 0 ? o.max_outer : 40;
        // measured crossover of the per-iteration cost on GB300 (Kuhn cubes):
        // the fused pass is ~30% faster at 35K nodes, equal near 250K, ~20%
        // slower at 900K (its larger vector traffic sits in the latency-bound
        // chunk pass)
        const bool solo = o.engine == PS_ENGINE_AUTO && m->solo && m->solo->fp32 && solo_ready(m);
        const bool fused = o.engine == PS_ENGINE_FUSED ||
                           (o.engine == PS_ENGINE_AUTO && m->dev.n_nodes <= kFusedMaxNodes);
        for (;;) {
            rc = true_residual(m, s, &rr);
            if (rc != PS_OK) break;
            ++outer;
            if (rr <= stop_abs2) { status = PS_OK; break; }
            if (used >= max_it || outer > max_outer) { status = PS_ENOTCONV; break; }
            const double scale = 1.0 / std::sqrt(rr);
            // inner reduction: itol, or only what the outer tolerance still
            // needs (with a factor 10 of margin) when that is less
            const double it_k = inner_reduction(itol, tol, bb, rr);
            if (solo) {
                rc = solo_run<float>(m, scale, it_k * it_k, max_it - used, m->dev.n_nodes > kFusedMaxNodes, spin, s);
                if (rc != PS_OK) break;
            } else if (fused) {
                const CG1Vec v = cg1_vec(m);
                k_cg1_init_state<<<1, 32, 0, s>>>(w.st, it_k * it_k, max_it - used);
                k_cg1_start<<<g3, kBlock, 0, s>>>(np, m->prep.sh_total, v, w.r64, scale);
                m->launches += 2;
            } else {
                Cg2Args<float> a = cg2_args<float>(m);
                CK(reset_shares(m, s));
                k_cg2_start<float><<<m->g3c, kBlock, 0, s>>>(m->dev, a, w.r64, scale, w.x32, it_k * it_k, 1,
                                                             max_it - used);
                m->launches += 1;
                if (a.halo) {
                    k_halo_gather<<<grid_for(m->prep.sh_total, m->ctx->sms), kBlock, 0, s>>>(
                        m->prep.sh_total, m->dev.sh_ids, a, 0);
                    m->launches += 1;
                }
            }
            if ((rc = cuda_status(cudaGetLastError())) != PS_OK) break;
            if (!solo && (rc = run_cg_until_done<float>(m, gi, jac, fused, s)) != PS_OK) break;
            RC(read_state(m, s, &h));
            if (solo) solo_end(*m->solo, h.done != 0, h.iters);
            if (solo && !h.done) { rc = PS_ETIMEOUT; break; }
            used += h.iters;
            if (h.status == kCgBreakdown) { status = PS_EBREAKDOWN; rc = PS_OK; break; }
            if (solo) continue;    // (the correction is added already)
            if (fused)
                k_cg1_correct<<<g3, kBlock, 0, s>>>(np, w.x64, cg1_vec(m), w.st, 1.0 / scale);
            else
                k_correct<<<g3, kBlock, 0, s>>>(np, w.x64, w.x32, 1.0 / scale);
            m->launches += 1;
            if ((rc = cuda_status(cudaGetLastError())) != PS_OK) break;
        }
    }
    m->dev = saved;
    if (rc == PS_ETIMEOUT) check_dev_err(m->ctx);
    if (rc != PS_OK) return rc;
    RC(check_dev_err(m->ctx));
    info->iters_outer = outer;
    info->iters_inner = used;
    info->rel_res = bb > 0 ? std::sqrt(rr / bb) : std::sqrt(rr);
    info->converged = status == PS_OK;
    info->status = status;
    return status;
}

}  // namespace ps

// ---------------------------------------------------------------- ABI: apply / solve
extern "C" int ps_pressure_apply(ps_mesh *m, const void *x, void *y, int prec, void *stream) {
    if (!m || !x || !y || (prec != PS_F32 && prec != PS_F64) || x == y) return PS_EINVAL;
    if (!m->coeff_ok) return PS_ESTATE;
    std::lock_guard<std::mutex> lk(m->ctx->mu);
    CK(cudaSetDevice(m->ctx->device));
    RC(ensure_workspace(m));
    cudaStream_t s = (cudaStream_t)stream;
    Workspace &w = m->ws;
    if (prec == PS_F32) return launch_apply<float>(m, (const float *)x, (float *)y, w.part32, s);
    return launch_apply<double>(m, (const double *)x, (double *)y, w.part64, s);
}

extern "C" void ps_solve_opts_default(ps_solve_opts *o) {
    if (!o) return;
    std::memset(o, 0, sizeof(*o));
    o->tol = 1e-10;
    o->max_iters = 100000;
    o->mode = PS_MODE_MIXED;
    o->precond = PS_PRECOND_JACOBI;
    o->inner_tol = 1e-4;
    o->max_outer = 40;
    o->graph_iters = 32;
    o->engine = PS_ENGINE_AUTO;
}

extern "C" int ps_pressure_solve(ps_mesh *m, const double *b, double *x, const ps_solve_opts *opts,
                                 ps_solve_info *info, void *stream) {
    if (!m || !b || !x) return PS_EINVAL;
    if (!m->coeff_ok) return PS_ESTATE;
    std::lock_guard<std::mutex> lk(m->ctx->mu);
    return ps::pressure_solve_locked(m, b, x, opts, info, (cudaStream_t)stream);
}

// ps_pressure_solve with the context mutex held by the caller.
int ps::pressure_solve_locked(ps_mesh *m, const double *b, double *x, const ps_solve_opts *opts,
                              ps_solve_info *info, cudaStream_t s) {
    ps_solve_opts o;
    if (opts) o = *opts; else ps_solve_opts_default(&o);
    if (o.mode != PS_MODE_FP64 && o.mode != PS_MODE_MIXED) return PS_EINVAL;
    if (o.engine < PS_ENGINE_AUTO || o.engine > PS_ENGINE_FUSED) return PS_EINVAL;
    ps_solve_info local;
    ps_solve_info *inf = info ? info : &local;
    std::memset(inf, 0, sizeof(*inf));
    auto t0 = std::chrono::steady_clock::now();
    CK(cudaSetDevice(m->ctx->device));
    if (o.mode == PS_MODE_MIXED && o.engine == PS_ENGINE_PERSISTENT && o.precond != PS_PRECOND_NONE) {
        ps_mesh *one[1] = {m};
        const double *bb[1] = {b};
        double *xx[1] = {x};
        int rc = batch_solve_locked(one, 1, bb, xx, o, inf, s);
        inf->seconds = std::chrono::duration<double>(std::chrono::steady_clock::now() - t0).count();
        return rc;
    }
    RC(ensure_workspace(m));
    Workspace &w = m->ws;
    const int64_t n = m->dev.n_nodes, nu = m->prep.n_nodes;   // unknowns, caller's vertices
    const int g = grid_for(n, m->ctx->sms), gu = grid_for(nu, m->ctx->sms);
    m->launches = 0;
    k_perm_in<double, double><<<g, kBlock, 0, s>>>(n, b, w.b64, m->d_old_of_new, m->dev.dirichlet);
    k_perm_in<double, double><<<g, kBlock, 0, s>>>(n, x, w.x64, m->d_old_of_new, m->dev.dirichlet);
    m->launches += 2;
    if (m->d_slave) {        // merged periodic vertices: their loads add onto the unknown
        k_add_slaves<<<g, kBlock, 0, s>>>(n, m->d_slave_ptr, m->d_slave, b, w.b64, m->dev.dirichlet);
        m->launches += 1;
    }
    CK(cudaGetLastError());
    int rc = solve_internal(m, o, inf, s);
    if (rc == PS_OK || rc == PS_ENOTCONV || rc == PS_EBREAKDOWN) {
        k_perm_out<double, double><<<gu, kBlock, 0, s>>>(nu, w.x64, x, m->d_new_of_old);
        m->launches += 1;
        CK(cudaGetLastError());
        CK(cudaStreamSynchronize(s));
    }
    inf->kernel_launches = m->launches;
    inf->seconds = std::chrono::duration<double>(std::chrono::steady_clock::now() - t0).count();
    return rc;
}

// ---------------------------------------------------------------- debug hooks (host only)
extern "C" int ps_debug_cg_apply(ps_mesh *m, const void *x, void *y, double *pap, void *stream) {
    if (!m || !x || !y || x == y) return PS_EINVAL;
    if (!m->coeff_ok) return PS_ESTATE;
    std::lock_guard<std::mutex> lk(m->ctx->mu);
    CK(cudaSetDevice(m->ctx->device));
    RC(ensure_workspace(m));
    cudaStream_t s = (cudaStream_t)stream;
    Workspace &w = m->ws;
    const int64_t n = m->dev.n_nodes, nu = m->prep.n_nodes;
    const int g = grid_for(n, m->ctx->sms), gu = grid_for(nu, m->ctx->sms);
    // p_old = x, r = 0 and beta = 1: the kernel's direction p = D^-1 r + beta p is x itself
    k_perm_in<float, float><<<g, kBlock, 0, s>>>(n, (const float *)x, w.p32, m->d_old_of_new, m->dev.dirichlet);
    CK(cudaMemsetAsync(w.r32, 0, m->dev.n_pad * sizeof(float), s));
    CgState hs;
    std::memset(&hs, 0, sizeof(hs));
    hs.beta = 1.0;
    hs.rz = 1.0;
    CK(cudaMemcpyAsync(w.st, &hs, sizeof(hs), cudaMemcpyHostToDevice, s));
    const Cg2Args<float> ca = cg2_args<float>(m);
    CK(reset_shares(m, s));
    if (ca.halo)
        k_halo_gather<<<grid_for(m->prep.sh_total, m->ctx->sms), kBlock, 0, s>>>(m->prep.sh_total,
                                                                                m->dev.sh_ids, ca, 0);
    launch_k1_f32(m, ca, s);
    VecArgs<float> va;
    std::memset(&va, 0, sizeof(va));
    va.y = w.q32;
    va.partial = w.part32;
    k_shared<float, kApply><<<m->grid2, kBlock, 0, s>>>(m->dev, va, 0);
    k_perm_out<float, float><<<gu, kBlock, 0, s>>>(nu, w.q32, (float *)y, m->d_new_of_old);
    CK(cudaGetLastError());
    CK(cudaMemcpyAsync(&hs, w.st, sizeof(hs), cudaMemcpyDeviceToHost, s));
    CK(cudaStreamSynchronize(s));
    int herr = 0;
    CK(cudaMemcpy(&herr, m->ctx->d_err, sizeof(int), cudaMemcpyDeviceToHost));
    if (herr) {
        cudaMemset(m->ctx->d_err, 0, sizeof(int));
        return PS_ETIMEOUT;
    }
    if (pap) *pap = hs.pq;
    return PS_OK;
}

extern "C" int ps_mesh_get_jacobi(const ps_mesh *m, int precision, void *dinv_host, void *stream) {
    if (!m || !dinv_host || (precision != PS_F32 && precision != PS_F64)) return PS_EINVAL;
    if (!m->coeff_ok) return PS_ESTATE;
    CK(cudaSetDevice(m->ctx->device));
    CK(cudaStreamSynchronize(reinterpret_cast<cudaStream_t>(stream)));
    const PrepMesh &p = m->prep;
    const size_t esz = precision == PS_F64 ? 8 : 4;
    std::vector<unsigned char> d(p.n_dofs * esz);
    const void *src = precision == PS_F64 ? (const void *)m->dev.dinv64 : (const void *)m->dev.dinv32;
    CK(cudaMemcpy(d.data(), src, d.size(), cudaMemcpyDeviceToHost));
    unsigned char *out = static_cast<unsigned char *>(dinv_host);
    for (int64_t j = 0; j < p.n_nodes; ++j) std::memcpy(out + j * esz, d.data() + (size_t)p.new_of_old[j] * esz, esz);
    return PS_OK;
}

extern "C" int ps_debug_prepare(int dim, int64_t n_nodes, const double *coords, int64_t n_elems,
                                const int32_t *conn, const uint8_t *dirichlet, const int32_t *periodic,
                                const ps_mesh_opts *opts, ps_mesh_stats *stats) {
    if (!coords || !conn) return PS_EINVAL;
    PrepOptions po;
    if (opts) {
        po.chunk_elems = opts->chunk_elems;
        po.chunk_nodes_max = opts->chunk_nodes_max;
        if (opts->split_lead < -1) return PS_EINVAL;
        po.split_lead = opts->split_lead > 0 ? opts->split_lead : 0;
    }
    po.periodic = periodic;
    PrepMesh pm;
    std::string err = prepare_mesh(dim, n_nodes, coords, n_elems, conn, dirichlet, po, pm);
    if (!err.empty()) {
        ps_set_last_error(err.c_str());
        return PS_EINVAL;
    }
    err = validate_prep(pm, conn);
    if (err.empty() && pm.max_loc <= 16383) {
        for (int stars : {kSoloStars, kSoloBatchStars}) {
            SoloPrep sp;
            build_solo(pm, 152, stars, sp);
            if (err.empty() && sp.max_loc <= 16383 && sp.max_star * kPatchSlots <= 65535) err = validate_solo(pm, sp);
        }
    }
    if (!err.empty()) {
        ps_set_last_error(err.c_str());
        return PS_ESTATE;
    }
    if (stats) {
        std::memset(stats, 0, sizeof(*stats));
        stats->n_nodes = pm.n_nodes;
        stats->n_elems = pm.n_elems;
        stats->n_free = pm.n_free;
        stats->dim = pm.dim;
        stats->n_chunks = pm.n_chunks;
        stats->n_shared = pm.n_shared;
        stats->chunk_node_refs = pm.loc_total;
        stats->max_chunk_elems = pm.max_elem;
        stats->max_chunk_nodes = pm.max_loc;
        SmemLayout l64 = make_layout(8, pm.max_loc, pm.max_patch, pm.max_inc);
        stats->reserved[0] = pm.n_patches;
        stats->reserved[1] = pm.inc_total;
        stats->device_bytes = l64.total;  // shared memory per block of the FP64 pass
    }
    return PS_OK;
}

// ---------------------------------------------------------------- kernel timing
extern "C" int ps_profile_kernel(ps_mesh *m, int which, int reps, void *stream, double *avg_ms) {
    if (!m || !avg_ms || reps < 1 || which < 0 || which > 6) return PS_EINVAL;
    if (!m->coeff_ok) return PS_ESTATE;
    std::lock_guard<std::mutex> lk(m->ctx->mu);
    CK(cudaSetDevice(m->ctx->device));
    RC(ensure_workspace(m));
    cudaStream_t s = (cudaStream_t)stream;
    Workspace &w = m->ws;
    MeshDev &d = m->dev;
    // a state that keeps every kernel running (done = 0, huge stop criterion unused)
    CgState hs;
    std::memset(&hs, 0, sizeof(hs));
    hs.rz = 1.0;
    hs.alpha = 0.0;
    hs.beta = 0.0;
    hs.max_iters = 1LL << 60;
    hs.stop_rr = -1.0;
    hs.first = 1;
    hs.free_run = 1;     // the fused pass never stops
    CK(cudaMemcpyAsync(w.st, &hs, sizeof(hs), cudaMemcpyHostToDevice, s));
    CK(reset_shares(m, s));
    // solves on chip leave the FP32 vectors untouched, and p.Ap = 0 would end
    // the run: any positive residual (0x3f3f3f3f = 0.747)
    if (m->solo && m->solo->fp32) {
        CK(cudaMemsetAsync(w.r32, 0x3f, (size_t)d.n_pad * 4, s));
        CK(cudaMemsetAsync(w.r32b, 0x3f, (size_t)d.n_pad * 4, s));
    }
    cudaEvent_t e0, e1;
    CK(cudaEventCreate(&e0));
    CK(cudaEventCreate(&e1));
    auto one = [&]() {
        switch (which) {
            case 0: {
                Cg2Args<float> a = cg2_args<float>(m);
                launch_k1_f32(m, a, s);
                break;
            }
            case 1: {
                Cg2Args<float> a = cg2_args<float>(m);
                k_cg2_update<float><<<m->g3c, kBlock, 0, s>>>(d, a);
                break;
            }
            case 2: {
                VecArgs<float> a;
                std::memset(&a, 0, sizeof(a));
                a.x = w.p32;
                a.y = w.q32;
                a.partial = w.part32;
                if (d.dim == 2) k_chunks<2, float, kApply><<<d.n_chunks, kBlock, d.sm32.total, s>>>(d, a);
                else k_chunks<3, float, kApply><<<d.n_chunks, kBlock, d.sm32.total, s>>>(d, a);
                k_shared<float, kApply><<<m->grid2, kBlock, 0, s>>>(d, a, d.n_chunks);
                break;
            }
            case 3: {
                VecArgs<double> a;
                std::memset(&a, 0, sizeof(a));
                a.x = w.x64;
                a.y = w.q64;
                a.b = w.b64;
                a.partial = w.part64;
                a.dotbuf = w.dot1;
                a.st = w.st;
                if (d.dim == 2) k_chunks<2, double, kResid><<<d.n_chunks, kBlock, d.sm64.total, s>>>(d, a);
                else k_chunks<3, double, kResid><<<d.n_chunks, kBlock, d.sm64.total, s>>>(d, a);
                break;
            }
            case 4: {
                Cg2Args<double> a = cg2_args<double>(m);
                if (d.dim == 2) k_cg2_chunks<2, double><<<d.n_chunks, kBlock, d.sm64.total, s>>>(d, a);
                else k_cg2_chunks<3, double><<<d.n_chunks, kBlock, d.sm64.total, s>>>(d, a);
                break;
            }
            case 5:
                launch_cg1(m, cg1_vec(m), s);
                break;
            case 6: {
                const Cg2Args<float> a = cg2_args<float>(m);
                // as in the iteration: the gather and, in the first block, the
                // update kernel's rz, rr reduction and the end of the iteration
                if (a.halo)
                    k_halo_gather<<<grid_for(m->prep.sh_total, m->ctx->sms) + 1, kBlock, 0, s>>>(m->prep.sh_total,
                                                                                            d.sh_ids, a, 1);
                break;
            }
        }
    };
    one();  // warm-up
    CK(cudaEventRecord(e0, s));
    for (int r = 0; r < reps; ++r) one();
    CK(cudaEventRecord(e1, s));
    CK(cudaGetLastError());
    CK(cudaEventSynchronize(e1));
    float ms = 0.f;
    CK(cudaEventElapsedTime(&ms, e0, e1));
    cudaEventDestroy(e0);
    cudaEventDestroy(e1);
    *avg_ms = (double)ms / reps;
    // leave a clean state for the next solve
    std::memset(&hs, 0, sizeof(hs));
    hs.done = 1;
    CK(cudaMemcpyAsync(w.st, &hs, sizeof(hs), cudaMemcpyHostToDevice, s));
    CK(cudaStreamSynchronize(s));
    return check_dev_err(m->ctx);
}

// ---------------------------------------------------------------- ABI: mass form
extern "C" int ps_mesh_set_mass(ps_mesh *m, int mass) {
    if (!m || (mass != PS_MASS_CONSISTENT && mass != PS_MASS_LUMPED)) return PS_EINVAL;
    std::lock_guard<std::mutex> lk(m->ctx->mu);
    CK(cudaSetDevice(m->ctx->device));
    const int lumped = mass == PS_MASS_LUMPED ? 1 : 0;
    if (m->dev.lumped == lumped) return PS_OK;
    m->dev.lumped = lumped;
    // captured solve graphs hold the mesh descriptor by value
    free_graphs(m);
    if (!m->coeff_ok) return PS_OK;
    RC(ensure_workspace(m));
    RC(ps::star_update_device(m, nullptr, 0.0, nullptr));
    CK(cudaDeviceSynchronize());
    return PS_OK;
}
