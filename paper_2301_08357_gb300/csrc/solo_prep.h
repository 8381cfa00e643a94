// Host layout of the on-chip CG of one mesh (solo.h).
#pragma once
#include <stdint.h>

#include <string>
#include <vector>

#include "mesh_prep.h"

namespace ps {

constexpr int kSoloMaxBlocks = 160;
// Stars per block of a mesh solved alone (larger meshes use every SM): fewer
// leave threads idle, more lengthen the FP64 pass (57 FP64 operations per star
// at two per clock and SM).
constexpr int kSoloStars = 64;
// Of a mesh in a batch, where the blocks of many meshes share the SMs: with the
// padding of the groups about two per thread, which stay in registers.  More
// are more per second but a longer iteration, and the meshes with the most
// iterations set the time (16 meshes, half 2D of up to 167,000 triangles: 320
// in 2D 6.0 ms, 448 5.3, 672 6.8; 896 in 3D 7.3).
constexpr int kSoloBatchStars = 448;

// One block's part of the mesh: a contiguous range of star groups and the
// unknowns they touch (interior: touched by this block alone; shared after
// them).
struct SoloBlock {
    int32_t star0, n_star;    // padded stars (multiples of kStarLanes)
    int32_t node0;            // first entry in gid
    int32_t n_int, n_loc;
    int32_t goff0, ell0;      // first entries in goff and ell
    int32_t n_ell;
    int32_t sh0;              // first entry in sh (n_loc - n_int of them)
};

// Host layout.  Contribution slot of star q, slot k: q * kPatchSlots + k.
struct SoloPrep {
    std::vector<SoloBlock> blocks;
    std::vector<uint32_t> ids;     // [patch_total * kStarIds] star ids in the block's node numbering (layout.h)
    std::vector<int32_t> gid;      // unknown of every local node
    // contribution slots of the nodes, 32 nodes at a time: words
    // [goff[g], goff[g + 1]) of group g hold, two slots per word, the lists of
    // nodes 32 g .. 32 g + 31 as rows of 32 words; lists are padded to the
    // group's longest with the block's zero slot (n_star * kPatchSlots)
    std::vector<uint32_t> goff;    // per block: one per group of 32 local nodes, and the end
    std::vector<uint32_t> ell;
    std::vector<int32_t> sh;       // [4 per shared local node] partials begin, end, own slot, 1 = owner
    int n_slots = 0;               // partial sums
    int max_star = 0, max_loc = 0, max_ell = 0, max_sh = 0;
};
void build_solo(const PrepMesh &m, int sms, int stars_per_block, SoloPrep &out);
// Checks what the kernel relies on: every star's ids name its unknowns in its
// block's numbering, every contribution is in the list of its node exactly
// once and all other entries are the zero slot, shared unknowns' partial slots
// are a bijection with one owner each.  "" or the first fault.
std::string validate_solo(const PrepMesh &m, const SoloPrep &s);

}  // namespace ps
