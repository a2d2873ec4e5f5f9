// What a grouped launch (group_gemm.cuh) carries, and the host rules that fill it and choose its form.  Plain C++: no device code.
#pragma once

#include <cstdint>
#include <algorithm>

#include "adapt_internal.h"

namespace adapt {

constexpr int kGroupMax = 64;           // entries per launch (the parameters stay below 4 KB)
constexpr int kGroupCluster = 4;        // CTAs per cluster of a launch with shared tiles

struct GroupItem {
    const unsigned short* A;
    const unsigned short* B;
    unsigned short* C;
    int M, N, K;
    int P_n;
    short pieces;                       // pieces of the k range; 0: CUDA-core tiles
    short share_log2;                   // CTAs that share a tile's pieces: 1, 2 or 4 (group_share)
    int k_per_piece;
    int tiles;                          // 64 x 64 tiles of one entry
    int tile_end;                       // CTAs of this and all earlier items: a tile each, or 2^share_log2 to a tile
};
struct GroupParams {
    int count;
    int ring;
    int prefetch;
    int dtype;
    int k_max;                          // largest K and most pieces of the list
    int pieces_max;
    int entries;                        // entries of an item (a strided batch; a list: 1)
    int sync_ctas;                      // the first CTAs, in clusters of kGroupCluster: those of shared tiles and what fills their last cluster
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
    it->pieces = simt ? 0 : (short)c.cluster;
    it->share_log2 = 0;
    it->k_per_piece = simt ? 0 : (int)round_up(ceil_div(s.K, c.cluster), 16);
    return simt ? 1 : it->pieces == 1 ? (int)ceil_div(s.K, 2 * kClusterKS) : (it->pieces / 2) * (int)ceil_div(it->k_per_piece, kClusterKS);
}

inline void group_clear(GroupParams& p)
{
    p.count = 0;
    p.ring = 1;
    p.k_max = 0;
    p.pieces_max = 0;
    p.entries = 1;
    p.sync_ctas = 0;
}
// Appends an item that stands for `entries` entries.  Items with shared tiles come first, those shared by more CTAs before the others; what
// follows them starts on a whole cluster.
inline void group_add(GroupParams& p, const GroupItem& it, int chain, int64_t entries = 1)
{
    int begin = p.count > 0 ? p.item[p.count - 1].tile_end : 0;
    if (it.share_log2 == 0 && p.sync_ctas % kGroupCluster) {
        begin = p.sync_ctas = (int)round_up(p.sync_ctas, kGroupCluster);
        p.item[p.count - 1].tile_end = begin;
    }
    p.item[p.count] = it;
    p.item[p.count].tile_end = (int)(entries * ((int64_t)it.tiles << it.share_log2) + begin);
    p.ring = std::max(p.ring, cluster_seq_ring(chain));
    p.k_max = std::max(p.k_max, it.K);
    p.pieces_max = std::max(p.pieces_max, (int)it.pieces);
    p.entries = (int)entries;
    if (it.share_log2 > 0) p.sync_ctas = p.item[p.count].tile_end;
    ++p.count;
}
// CTAs of the launch: whole clusters where there are any.
inline int group_grid(GroupParams& p)
{
    if (p.sync_ctas == 0) return p.item[p.count - 1].tile_end;
    p.sync_ctas = (int)round_up(p.sync_ctas, kGroupCluster);
    return (int)round_up(std::max(p.item[p.count - 1].tile_end, p.sync_ctas), kGroupCluster);
}

// What CTA `cta` of the launch computes: tile `tile` of an entry of an item, as the q-th of the CTAs that share it; false: nothing.
struct GroupPlace { int item, entry, tile, q; };
ADAPT_HOST_DEVICE bool group_place(const GroupParams& p, int cta, GroupPlace& w)
{
    int lo = 0, hi = p.count - 1;                           // the first item whose CTAs end beyond this one
    while (lo < hi) {
        const int mid = (lo + hi) >> 1;
        if (cta < p.item[mid].tile_end) hi = mid; else lo = mid + 1;
    }
    const GroupItem& it = p.item[lo];
    const int local = cta - (lo > 0 ? p.item[lo - 1].tile_end : 0), unit = local >> it.share_log2;
    w.item = lo;
    w.q = local & ((1 << it.share_log2) - 1);
    w.entry = unit < it.tiles ? 0 : unit / it.tiles;
    w.tile = unit - w.entry * it.tiles;
    return cta < it.tile_end && w.entry < p.entries;
}

// An entry of a list, and the stages one group of warps of its tiles walks.
struct GroupEntry { GroupItem item; int chain; };

// Shares the tiles of an entry whose chain the launch would wait for between two CTAs (four pieces) or four (eight, sixteen), whose groups of
// warps then walk one piece each, or two.
inline void group_share(GroupEntry* e, double average_chain)
{
    GroupItem& it = e->item;
    if (it.pieces < 4 || e->chain < 3 || 2 * e->chain <= average_chain) return;
    it.share_log2 = it.pieces == 4 ? 1 : 2;
    e->chain = it.pieces / (2 << it.share_log2) * (int)ceil_div(it.k_per_piece, kClusterKS);
}

// The order of a list's entries in the launch.  An unaligned stage takes a group of warps 1.4 us, so the tile with the most of them is what a
// short list waits for: its tiles are shared where the chain is longer than half of what a CTA slot (two per SM) has to do on average and
// the list stays within four CTAs per SM.  Beyond, the SMs are busy while the long chains run (the longest come first), and clusters, which
// start when four slots of a GPC are free, cost more than they save: 8 layers of 16 .. 1024 a side 9.7 -> 7.7 us, 24 layers 19.3 -> 11.8,
// 15 layers with K > 256 19.4 -> 17.5, but 47 layers (1018 CTAs shared, 762 not) 20.9 -> 27.3.
inline void group_order(GroupEntry* e, size_t n, int n_sm)
{
    double work = 0.0;
    for (size_t j = 0; j < n; ++j) work += (double)e[j].item.tiles * e[j].chain;
    int64_t ctas = 0;
    GroupEntry as_is[kGroupMax];
    for (size_t j = 0; j < n; ++j) {
        as_is[j] = e[j];
        group_share(&e[j], work / (2.0 * n_sm));
        ctas += (int64_t)e[j].item.tiles << e[j].item.share_log2;
    }
    if (ctas > 4 * (int64_t)n_sm) std::copy(as_is, as_is + n, e);
    std::stable_sort(e, e + n, [](const GroupEntry& x, const GroupEntry& y) {
        return x.item.share_log2 != y.item.share_log2 ? x.item.share_log2 > y.item.share_log2 : x.chain > y.chain;
    });
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
