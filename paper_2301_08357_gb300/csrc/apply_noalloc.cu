// ps_pressure_apply_noalloc: the operator apply y = A x without any device
// allocation.
//
// Who needs it: callers that cannot call cudaMalloc at the point where they
// apply the operator -- for example a host framework whose caching allocator
// has already reserved the device memory it is allowed to use (a fresh
// cudaMalloc would fail or push it over its budget), or a solver loop that
// must not let an allocation implicitly synchronise the device between time
// steps.  ps_pressure_apply allocates the mesh's solver workspace (its scratch
// among it: partial sums of shared nodes) on first use; this variant instead
// carves that scratch out of one file-scope __device__ array, which every GPU that
// loads the library holds until the process exits.
//
// The array's host-side name is only a stand-in; the device address is looked
// up once per device with cudaGetSymbolAddress (that device current) when a
// context is created on it (ps_ctx_create calls noalloc_setup): the lookup
// loads this file's module, which commits the array's device memory then and
// not inside a later apply.  The cached address assumes the device's primary
// context lives until the process exits (no cudaDeviceReset in between).
// Every call shares the array and it keeps the last call's contents; nothing
// in it needs to start at zero because a call that completes writes every
// entry it later reads.  (If a bounded device wait gives up, the kernel
// leaves its chunk unwritten: y is then undefined, and the context's error
// flag reports PS_ETIMEOUT at its next synchronising call.)  Calls whose work
// overlaps on the GPU (different streams, or different meshes at the same
// time) race on it.
#include <cuda_runtime.h>

#include <cstring>
#include <mutex>

#include "../../include/pressure.h"
#include "internal.h"

using namespace ps;

namespace {

constexpr size_t kScratchBytes = size_t(16) << 20;   // 16 MiB
constexpr int kMaxDevices = 64;

static __device__ __align__(256) unsigned char g_noalloc_scratch[kScratchBytes];

std::mutex g_mu;
void *g_addr[kMaxDevices] = {nullptr};

size_t align256(size_t v) { return (v + 255) / 256 * 256; }

// Device address of the scratch array on `device` (which must be current).
int scratch_address(int device, void **out) {
    if (device < 0 || device >= kMaxDevices) return PS_EINVAL;
    std::lock_guard<std::mutex> lk(g_mu);
    if (!g_addr[device]) {
        void *p = nullptr;
        cudaError_t e = cudaGetSymbolAddress(&p, g_noalloc_scratch);
        if (e != cudaSuccess || p == nullptr) {
            ps_set_last_error(e == cudaSuccess ? "no device address for the allocation-free scratch"
                                               : cudaGetErrorString(e));
            cudaGetLastError();
            return e == cudaErrorMemoryAllocation ? PS_ENOMEM : PS_ECUDA;
        }
        g_addr[device] = p;
    }
    *out = g_addr[device];
    return PS_OK;
}

}  // namespace

// Called by ps_ctx_create with `device` current: looks the scratch array up
// (loading this module and committing its memory) once per device.
int ps::noalloc_setup(int device) {
    void *p = nullptr;
    return scratch_address(device, &p);
}

extern "C" int ps_pressure_apply_noalloc(ps_mesh *m, const void *x, void *y, int prec, void *stream) {
    if (!m || !x || !y || (prec != PS_F32 && prec != PS_F64) || x == y) return PS_EINVAL;
    if (!m->coeff_ok) return PS_ESTATE;
    const size_t esz = prec == PS_F32 ? 4 : 8;
    const int64_t np = m->dev.n_pad;
    const int64_t sh = m->prep.sh_total > 0 ? m->prep.sh_total : 1;
    // the documented limit: room for permuted copies of x and y beside the
    // partial sums (only the latter are used: the kernels read x and write y
    // in the caller's numbering)
    const size_t need = 2 * align256((size_t)np * esz) + align256((size_t)sh * esz);
    if (need > kScratchBytes) {
        char msg[160];
        snprintf(msg, sizeof(msg),
                 "mesh too large for ps_pressure_apply_noalloc: needs %zu bytes of scratch, limit %zu",
                 need, kScratchBytes);
        ps_set_last_error(msg);
        return PS_EINVAL;
    }
    std::lock_guard<std::mutex> lk(m->ctx->mu);
    cudaError_t e = cudaSetDevice(m->ctx->device);
    if (e != cudaSuccess) {
        ps_set_last_error(cudaGetErrorString(e));
        return PS_ECUDA;
    }
    void *base = nullptr;
    int rc = scratch_address(m->ctx->device, &base);
    if (rc != PS_OK) return rc;
    cudaStream_t s = (cudaStream_t)stream;
    if (prec == PS_F32) return launch_apply<float>(m, (const float *)x, (float *)y, (float *)base, s);
    return launch_apply<double>(m, (const double *)x, (double *)y, (double *)base, s);
}
