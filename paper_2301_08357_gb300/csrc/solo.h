// On-chip CG of one mesh (solo.cu): the inner solve of ps_pressure_solve in
// one cooperative kernel whose blocks keep their part of every CG vector in
// shared memory from the first iteration to the last.
#pragma once
#include "ops.cuh"
#include "solo_prep.h"

struct ps_mesh;

namespace ps {

struct BatchPlan;
struct DevAlloc;

// Offsets of a block's arrays in shared memory.
struct SoloSmem {
    uint32_t val, r, s, p, x, di, m, w, contrib, goff, ell, sh, total;
};

// Device copy, owned by the mesh (null: the mesh does not fit).
struct Solo {
    int n_blocks = 0, n_slots = 0, mean_star = 0;
    int threads = 0;               // FP32 kernels (the FP64 one: at most 256)
    SoloBlock *blocks = nullptr;
    uint4 *ids4 = nullptr;
    uint32_t *ids1 = nullptr;
    int32_t *gid = nullptr;
    uint32_t *goff = nullptr, *ell = nullptr;
    int4 *sh = nullptr;
    SoloSmem sm32, sm64;
    bool fp32 = false, fp64 = false;   // which precisions fit
    // workspace, allocated by the first solve
    void *part = nullptr;              // partial sums, two buffers of tagged words
    uint4 *exch = nullptr;             // dot-product shares, two buffers of tagged words
    uint32_t tag = 0;                  // last tag used (0: the words are to be cleared)
};

int solo_set_attrs();
int solo_upload(ps_mesh *m);
void solo_release(ps_mesh *m);
// The workspace of the mesh's runs, allocated on first use; false: the context
// has no room for it (the solve then takes the kernels that need none).
bool solo_ready(ps_mesh *m);

// ---- the FP32 kernel over a batch: blocks of many meshes side by side.
// Layout of a mesh in a batch (its arrays go to `owner`; the mesh's own layout
// when that has the same blocks), or null: the mesh does not fit, the batch
// runs it chunk by chunk.
int solo_batch_layout(ps_mesh *m, std::vector<DevAlloc> &owner, Solo **out);
// The mesh's size is one of those that get a layout of their own there.
bool solo_batch_size(const ps_mesh *m);
// One cooperative launch: its thread blocks run the meshes' blocks that are
// theirs in the plan's list, one after another.
struct SoloLaunch {
    int first, blocks, threads;   // first entry of the list's pointers
    uint32_t smem;
};
// Places the blocks of the plan's meshes that have a layout and uploads what
// the launches read; a launch takes its runs to their end.
int solo_plan_build(BatchPlan &plan, cudaStream_t s);
int solo_plan_enqueue(BatchPlan &plan, cudaStream_t s);
// Clears the plan's exchanged words (before tags run out, after a wait's limit).
int solo_plan_clear(BatchPlan &plan, cudaStream_t s);
// One inner run from the residual r64 (times scale) in the mesh's workspace:
// x64 += the correction found / scale; the CG state receives the iteration
// count and status.  T = float: relative reduction tol2 of r.r; double: stop
// at r.r <= tol2.  spin_limit: polls of a wait (ps_solve_opts.grid_spin_limit).
template <typename T>
int solo_run(ps_mesh *m, double scale, double tol2, long long max_iters, bool nan_breaks, uint32_t spin_limit,
             cudaStream_t s);
// After the run's state is on the host: iters of it (done) or no end (a wait
// gave up).
inline void solo_end(Solo &S, bool done, long long iters) { S.tag = done ? S.tag + (uint32_t)iters + 2u : 0u; }

}  // namespace ps
