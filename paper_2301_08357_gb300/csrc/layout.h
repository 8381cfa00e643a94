// Device data layout of one preprocessed mesh, shared by the host
// preprocessing (mesh_prep.cpp) and the CUDA kernels.
//
// Elements are partitioned into "chunks" of consecutive elements along a Morton
// curve of their centroids, and inside a chunk into star-shaped patches.  Nodes touched by exactly one chunk are that
// chunk's interior nodes; they are numbered contiguously per chunk, so the
// chunk owns their rows outright.  Nodes touched by several chunks ("shared")
// are numbered after all interior nodes.  A chunk computes its element
// contributions in shared memory, sums them per local node through a fixed
// incidence list (deterministic, no atomics), writes its interior rows
// directly and writes one partial sum per shared local node, into a
// shared-node-major array (the partials of one shared node are contiguous); a
// second pass adds the partial sums of every shared node in chunk order.
//
// Every per-chunk segment starts on a 16-byte boundary so that it can be moved
// into shared memory with one cp.async.bulk copy.
#pragma once
#include <stdint.h>

namespace ps {

constexpr int kPatchMax = 6;     // elements per patch (star) at most
constexpr int kPatchIds = 12;    // u16 per patch record: m, a, b, ring[0..m], padding
constexpr int kPatchSlots = 9;   // contribution slots per patch: a, b, ring[0..6]
// FP64 element geometry per patch slot: 3D G_AB, G_A0, G_A1, G_B0, G_B1, G_01, |det|;
// 2D G_A0, G_A1, G_01, |det| (G_ab = c_a.c_b / (d! |det|), c_a the cofactor vectors).
// Read when the star weights are formed; word k of element j of a patch lies
// at row j * W + k of its group of 32 patches (kStarLanes).
template <int D>
constexpr int kGeoWords = D == 3 ? 7 : 4;
constexpr int kPatchPad = 32;    // patch segments padded to whole groups (kStarLanes)
constexpr int kIncPad = 8;       // incidence segments padded to 8 u16
constexpr int kIncpPad = 8;      // incidence-pointer segments padded to 8 u16
constexpr int kShPad = 4;        // shared-id segments padded to 4 int32
constexpr int kMaxChunkPatches = 65535 / kPatchSlots;  // slot ids fit in u16
constexpr int kChunkThreads = 256;  // threads of a block that processes a chunk

// Elements of a chunk are grouped into "patches": the elements around one
// pivot (an edge (a, b) in 3D, a vertex a in 2D), ordered so that element j of
// the patch is (a, b, ring[j], ring[j+1]) in 3D and (a, ring[j], ring[j+1]) in
// 2D, j = 0..m-1.  A closed star repeats ring[0] as ring[m].  An element that
// joins no star is a patch of one (m = 1).  Patch record (u16): [0] = m,
// [1] = a, [2] = b (3D), [3 + j] = ring[j], j = 0..m; all local node ids.
// Contribution slots: 0 -> a, 1 -> b, 2 + j -> ring[j].

// Star weights.  Every operator pass evaluates a patch as one macro element:
// the sum of its elements' matrices, stored by its edges.  With A^s that sum
// and m_i = sum_j A^s_ij its row sums (the stiffness part has none, so m_i is
// the mass of the row: int alpha_h phi_i over the patch),
//     (A^s v)_i = sum_{j != i} A^s_ij (v_j - v_i) + m_i v_i,
// so an edge costs one difference and two multiply-adds whatever the number
// of elements around it, and a constant v meets no cancellation.  The m_i are
// summed over the chunk once and kept per local node (mrow).  A closed star
// (ring[m] = ring[0]) has nr = m ring nodes, an open one nr = m + 1.
// Patches are stored in groups of 32 (every chunk padded to whole groups), 16
// bytes per lane and row, so that a warp reads a row with one 512-byte load
// and every row lies at a constant offset from the patch's first:
//   FP32 record, rows of four words: words 0..4 the ids, 5.. the weights; six
//           rows hold a star of up to six ring nodes, a 3D mesh with an open
//           star of six has seven (kStarVec; MeshDev::srows)
//   FP64 weights, kStarVec64 rows of two
//   ids: a | b << 16, r0 | r1 << 16, r2 | r3 << 16, r4 | r5 << 16,
//           r6 | nr << 16 | closed << 20; node ids times 4, the byte offset of an
//           FP32 value (an uploaded chunk has fewer than 16,384 nodes)
//   weights, 3D: ab, (r_{nr-1}, r_0) (0 on an open star), (a, r_0), (b, r_0),
//           then for j = 1..nr-1: (a, r_j), (b, r_j), (r_{j-1}, r_j)
//   weights, 2D: (r_{nr-1}, r_0), (a, r_0), then for j = 1..nr-1: (a, r_j),
//           (r_{j-1}, r_j)
constexpr int kStarIds = 5;
constexpr int kStarRing = kPatchMax + 1;
constexpr int kStarLanes = 32;
template <int D>
constexpr int kStarW = D == 3 ? 22 : 14;                              // weights of an open star of six
template <int D>
constexpr int kStarVec = (kStarIds + kStarW<D> + 3) / 4;              // 7, 5
template <int D>
constexpr int kStarVec64 = kStarW<D> / 2;                             // 11, 7

struct ChunkDesc {
    int32_t patch_off;  // first (padded) patch of the chunk
    int32_t n_patch;
    int32_t node_off;   // first entry of the chunk's node block
    int32_t n_loc;      // local nodes = n_int + n_sh
    int32_t n_int;      // interior nodes: local 0..n_int-1 = new ids int_begin + l
    int32_t int_begin;
    int32_t sh_off;     // first entry in sh_ids / partial slots (padded)
    int32_t n_sh;       // shared local nodes: local n_int + j -> sh_ids[sh_off + j]
    int32_t incp_off;   // first entry of the chunk's incidence pointers (padded)
    int32_t inc_off;    // first entry of the chunk's incidence list (padded)
    int32_t n_inc;      // incidence entries (patch * kPatchSlots + slot)
    int32_t n_elem;
};
static_assert(sizeof(ChunkDesc) == 48, "ChunkDesc layout");

inline int64_t round_up(int64_t v, int64_t m) { return (v + m - 1) / m * m; }

}  // namespace ps
