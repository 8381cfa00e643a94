// Host layout of the on-chip CG (solo.h): star groups to blocks, the unknowns
// each block touches, its incidence lists and the partial-sum slots of shared
// unknowns.
#include <algorithm>

#include "solo_prep.h"

namespace ps {

void build_solo(const PrepMesh &m, int sms, int stars, SoloPrep &o) {
    o = SoloPrep();
    const int n_groups = (int)(m.patch_total / kStarLanes);
    sms = std::min(sms, kSoloMaxBlocks);
    const int64_t G = std::max<int64_t>(1, std::min<int64_t>(sms, (m.n_patches + stars - 1) / stars));
    // groups -> blocks by real stars
    std::vector<int> chunk_of(n_groups, 0), real(n_groups, 0);
    for (int c = 0; c < m.n_chunks; ++c)
        for (int q = 0; q < m.chunks[c].n_patch; ++q) {
            const int g = (m.chunks[c].patch_off + q) / kStarLanes;
            chunk_of[g] = c;
            real[g]++;
        }
    std::vector<int> first;   // first group of every block
    int64_t done = 0;
    for (int g = 0; g < n_groups; ++g) {
        if (first.empty() || done >= (int64_t)first.size() * m.n_patches / G) first.push_back(g);
        done += real[g];
    }
    first.push_back(n_groups);
    const int nb = (int)first.size() - 1;
    // unknowns touched by one block, or by several
    auto each = [&](int g, auto &&fn) {   // star index, patch record, chunk
        const ChunkDesc &cd = m.chunks[chunk_of[g]];
        for (int s = g * kStarLanes; s < (g + 1) * kStarLanes && s < cd.patch_off + cd.n_patch; ++s)
            fn(s, &m.pids[(size_t)s * kPatchIds], cd);
    };
    auto slots = [&](const uint16_t *rec, auto &&fn) {   // chunk-local node, slot
        const int pm = rec[0];
        const int nr = pm >= 2 && rec[3 + pm] == rec[3] ? pm : pm + 1;
        fn(rec[1], 0);
        if (m.dim == 3) fn(rec[2], 1);
        for (int j = 0; j < nr; ++j) fn(rec[3 + j], 2 + j);
    };
    std::vector<int32_t> last(m.n_dofs, -1), loc(m.n_dofs, -1), cnt(m.n_dofs, 0);
    for (int b = 0; b < nb; ++b)
        for (int g = first[b]; g < first[b + 1]; ++g)
            each(g, [&](int, const uint16_t *rec, const ChunkDesc &cd) {
                slots(rec, [&](int l, int) {
                    const int32_t u = m.loc_node[cd.node_off + l];
                    if (last[u] != b) {
                        last[u] = b;
                        cnt[u]++;
                    }
                });
            });
    std::vector<int32_t> base(m.n_dofs, 0), fill(m.n_dofs, 0);
    for (int64_t u = 0; u < m.n_dofs; ++u)
        if (cnt[u] > 1) {
            base[u] = o.n_slots;
            o.n_slots += cnt[u];
        }
    o.ids.assign((size_t)m.patch_total * kStarIds, 0);
    std::vector<int32_t> nodes;
    std::vector<int> deg;
    for (int b = 0; b < nb; ++b) {
        SoloBlock B;
        B.star0 = first[b] * kStarLanes;
        B.n_star = (first[b + 1] - first[b]) * kStarLanes;
        B.node0 = (int32_t)o.gid.size();
        nodes.clear();
        deg.clear();
        for (int g = first[b]; g < first[b + 1]; ++g)
            each(g, [&](int, const uint16_t *rec, const ChunkDesc &cd) {
                slots(rec, [&](int l, int) {
                    const int32_t u = m.loc_node[cd.node_off + l];
                    if (loc[u] < 0) {
                        loc[u] = (int32_t)nodes.size();
                        nodes.push_back(u);
                        deg.push_back(0);
                    }
                    deg[loc[u]]++;
                });
            });
        // interior first, then shared, each by the number of contributions
        // (the threads of a warp then sum lists of nearly the same length)
        std::vector<int32_t> order(nodes.size());
        for (size_t k = 0; k < order.size(); ++k) order[k] = (int32_t)k;
        std::stable_sort(order.begin(), order.end(), [&](int32_t x, int32_t y) {
            const bool sx = cnt[nodes[x]] > 1, sy = cnt[nodes[y]] > 1;
            if (sx != sy) return sy;
            if (deg[x] != deg[y]) return deg[x] > deg[y];
            return sx && nodes[x] < nodes[y];
        });
        B.n_loc = (int32_t)order.size();
        B.n_int = 0;
        B.goff0 = (int32_t)o.goff.size();
        B.ell0 = (int32_t)o.ell.size();
        B.sh0 = (int32_t)(o.sh.size() / 4);
        for (int k = 0; k < B.n_loc; ++k) {
            const int32_t u = nodes[order[k]];
            loc[u] = k;
            o.gid.push_back(u);
            if (cnt[u] == 1) {
                B.n_int++;
            } else {
                o.sh.insert(o.sh.end(), {base[u], base[u] + cnt[u], base[u] + fill[u], fill[u] == 0 ? 1 : 0});
                fill[u]++;
            }
        }
        const uint32_t zero = (uint32_t)(B.n_star * kPatchSlots) & 0xffffu;
        o.goff.push_back(0);
        for (int k0 = 0; k0 < B.n_loc; k0 += 32) {
            int longest = 0;
            for (int k = k0; k < std::min(k0 + 32, B.n_loc); ++k) longest = std::max(longest, deg[order[k]]);
            o.goff.push_back(o.goff.back() + (uint32_t)(longest + 1) / 2 * 32);
        }
        B.n_ell = (int32_t)o.goff.back();
        o.ell.resize((size_t)B.ell0 + B.n_ell, zero | zero << 16);
        std::vector<int> put(B.n_loc, 0);
        for (int g = first[b]; g < first[b + 1]; ++g)
            each(g, [&](int s, const uint16_t *rec, const ChunkDesc &cd) {
                uint32_t id[2 * kStarIds] = {0};
                slots(rec, [&](int l, int slot) {
                    const int32_t k = loc[m.loc_node[cd.node_off + l]];
                    uint32_t &w = o.ell[(size_t)B.ell0 + o.goff[(size_t)B.goff0 + k / 32] + put[k] / 2 * 32 + k % 32];
                    const uint32_t c = (uint32_t)((s - B.star0) * kPatchSlots + slot) & 0xffffu;
                    w = put[k] & 1 ? (w & 0xffffu) | c << 16 : (w & 0xffff0000u) | c;
                    put[k]++;
                    id[slot] = (4u * (uint32_t)k) & 0xffffu;
                });
                id[2 * kStarIds - 1] = m.sids[(size_t)s * kStarIds + kStarIds - 1] >> 16;
                for (int k = 0; k < kStarIds; ++k) o.ids[(size_t)s * kStarIds + k] = id[2 * k] | id[2 * k + 1] << 16;
            });
        for (int32_t u : nodes) loc[u] = -1;
        o.max_star = std::max(o.max_star, B.n_star);
        o.max_loc = std::max(o.max_loc, B.n_loc);
        o.max_ell = std::max(o.max_ell, B.n_ell);
        o.max_sh = std::max(o.max_sh, B.n_loc - B.n_int);
        o.blocks.push_back(B);
    }
}

std::string validate_solo(const PrepMesh &m, const SoloPrep &o) {
    std::vector<int> seen(m.patch_total, 0), slot(o.n_slots, 0), holders(m.n_dofs, 0), owners(m.n_dofs, 0);
    std::vector<int> chunk_of(m.patch_total, -1);
    for (int c = 0; c < m.n_chunks; ++c)
        for (int q = 0; q < m.chunks[c].n_patch; ++q) chunk_of[m.chunks[c].patch_off + q] = c;
    for (const SoloBlock &B : o.blocks) {
        if (B.star0 % kStarLanes || B.n_star % kStarLanes || B.n_loc > 16383 || B.n_star * kPatchSlots > 65535)
            continue;   // (a mesh of such blocks is not taken)
        std::vector<int> node_of((size_t)B.n_star * kPatchSlots, -1), hits(node_of.size(), 0);
        for (int l = 0; l < B.n_loc; ++l) holders[o.gid[B.node0 + l]]++;
        for (int q = 0; q < B.n_star; ++q) {
            const int s = B.star0 + q;
            seen[s]++;
            const uint32_t *w = &o.ids[(size_t)s * kStarIds];
            if (chunk_of[s] < 0) {
                if (w[4] >> 16) return "solo: pad star with ring nodes";
                continue;
            }
            const uint16_t *rec = &m.pids[(size_t)s * kPatchIds];
            const int nr = (int)((w[4] >> 16) & 7u);
            const bool closed = (w[4] >> 20) & 1u;
            if (nr != (closed ? rec[0] : rec[0] + 1)) return "solo: ring size";
            auto check = [&](int k, int local) {
                const uint32_t id = k & 1 ? w[k / 2] >> 16 : w[k / 2] & 0xffffu;
                if (id % 4 || (int)(id / 4) >= B.n_loc) return false;
                node_of[(size_t)q * kPatchSlots + k] = (int)(id / 4);
                return o.gid[B.node0 + id / 4] == m.loc_node[m.chunks[chunk_of[s]].node_off + local];
            };
            if (!check(0, rec[1]) || (m.dim == 3 && !check(1, rec[2]))) return "solo: pivot id";
            for (int j = 0; j < nr; ++j)
                if (!check(2 + j, rec[3 + j])) return "solo: ring id";
        }
        const uint32_t zero = (uint32_t)(B.n_star * kPatchSlots);
        for (int g = 0; g * 32 < B.n_loc; ++g)
            for (uint32_t k = o.goff[B.goff0 + g]; k < o.goff[B.goff0 + g + 1]; ++k) {
                if ((int)k >= B.n_ell) return "solo: list out of range";
                for (int h = 0; h < 2; ++h) {
                    const uint32_t c = (o.ell[(size_t)B.ell0 + k] >> (16 * h)) & 0xffffu;
                    if (c == zero) continue;
                    const int l = g * 32 + (int)(k % 32);
                    if (c > zero || l >= B.n_loc || node_of[c] != l) return "solo: contribution of another node";
                    hits[c]++;
                }
            }
        for (size_t c = 0; c < hits.size(); ++c)
            if (hits[c] != (node_of[c] >= 0 ? 1 : 0)) return "solo: contribution not summed exactly once";
        for (int l = B.n_int; l < B.n_loc; ++l) {
            const int32_t *si = &o.sh[4 * ((size_t)B.sh0 + l - B.n_int)];
            if (si[2] < si[0] || si[2] >= si[1] || si[0] < 0 || si[1] > o.n_slots) return "solo: partial slot";
            slot[si[2]]++;
            owners[o.gid[B.node0 + l]] += si[3];
        }
    }
    for (int64_t s = 0; s < m.patch_total; ++s)
        if (seen[s] != 1) return "solo: star not in exactly one block";
    for (int v : slot)
        if (v != 1) return "solo: partial slots not a bijection";
    for (int64_t u = 0; u < m.n_dofs; ++u)
        if (holders[u] < 1 || owners[u] != (holders[u] > 1 ? 1 : 0)) return "solo: unknown without exactly one owner";
    return "";
}

}  // namespace ps
