// What a grouped launch (group_gemm.cuh) carries, and the host rules that fill it and choose its form.  Plain C++: no device code.
#pragma once

#include <cstdint>
#include <algorithm>

#include "adapt_internal.h"

namespace adapt {

constexpr int kGroupMax = 64;           // entries per launch (the parameters stay below 4 KB)

struct GroupItem {
    const unsigned short* A;
    const unsigned short* B;
    unsigned short* C;
    int M, N, K;
    int P_n;
    int pieces;                         // pieces of the k range; 0: CUDA-core tiles
    int k_per_piece;
    int tiles;                          // 64 x 64 tiles of one entry
    int tile_end;                       // tiles of this and all earlier items
};
struct GroupParams {
    int count;
    int ring;
    int prefetch;
    int dtype;
    int k_max;                          // largest K and most pieces of the list
    int pieces_max;
    int64_t sa, sb, sc;                 // strided batch: item 0 stands for all entries, sa, sb, sc elements apart
    GroupItem item[kGroupMax];
};
static_assert(sizeof(GroupParams) <= 4096, "kernel parameters");

// Can an entry with this configuration run in the grouped launch?  The cluster kernel's tiles: the k range must not be a long
// chain (24 stages are about 10 us).  CUDA-core tiles: no k split and a few steps.
inline bool group_eligible(const Shape& s, const Config& c)
{
    if (c.family == ADAPT_FAM_SIMT) return c.P_k == 1 && s.K <= 64 && (int64_t)c.P_m * c.P_n <= 512;
    return c.family == ADAPT_FAM_CLUSTER && c.cluster * ceil_div(round_up(ceil_div(s.K, c.cluster), 16), kClusterKS) <= 24;
}

// Fills everything of an item but tile_end; returns its chain: the stages one group of warps of a tile walks.
inline int group_item(const Shape& s, const Config& c, const void* A, const void* B, void* C, GroupItem* it)
{
    it->A = (const unsigned short*)A;
    it->B = (const unsigned short*)B;
    it->C = (unsigned short*)C;
    it->M = (int)s.M; it->N = (int)s.N; it->K = (int)s.K;
    it->P_n = c.P_n;
    it->tiles = c.P_m * c.P_n;
    const bool simt = c.family == ADAPT_FAM_SIMT;
    it->pieces = simt ? 0 : c.cluster;
    it->k_per_piece = simt ? 0 : (int)round_up(ceil_div(s.K, c.cluster), 16);
    return simt ? 1 : it->pieces == 1 ? (int)ceil_div(s.K, 2 * kClusterKS) : (it->pieces / 2) * (int)ceil_div(it->k_per_piece, kClusterKS);
}

inline void group_clear(GroupParams& p)
{
    p.count = 0;
    p.ring = 1;
    p.k_max = 0;
    p.pieces_max = 0;
}
// Appends an item that stands for `entries` entries.
inline void group_add(GroupParams& p, const GroupItem& it, int chain, int64_t entries = 1)
{
    p.item[p.count] = it;
    p.item[p.count].tile_end = (int)(entries * it.tiles + (p.count > 0 ? p.item[p.count - 1].tile_end : 0));
    p.ring = std::max(p.ring, cluster_seq_ring(chain));
    p.k_max = std::max(p.k_max, it.K);
    p.pieces_max = std::max(p.pieces_max, it.pieces);
    ++p.count;
}

// The kernel of a launch: one stage with all warps on it (SHORT), or two groups of warps with a ring each.  SHORT is the body of a
// cluster's CTA: it multiplies one piece of the k range.  The CTAs of this launch are in no cluster, so an entry whose plan cuts a
// short k range into pieces (a plan table may name such a configuration) needs the other kernel, which walks all pieces.
struct GroupForm { bool short_k; int smem_bytes; };
inline GroupForm group_form(const GroupParams& p)
{
    GroupForm f;
    f.short_k = p.k_max <= kClusterKS && p.pieces_max <= 1;
    f.smem_bytes = f.short_k ? cluster_smem_bytes(1) : cluster_seq_smem_bytes(p.ring);
    return f;
}

}  // namespace adapt
