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

// What sharing the tiles of a list is weighed with (us): a stage of a group of warps on aligned rows, what the shift of an operand adds whose rows are
// not on 16-byte boundaries (a whole tile's rows of it), the rest of a CTA's life, the exchange of a shared tile, and a round of further CTAs (two per SM).
constexpr double kGroupStageUs = 0.5, kGroupShiftUs = 0.4, kGroupTileUs = 1.5, kGroupExchangeUs = 0.3, kGroupRoundUs = 3.5;

// An entry of a list, and the stages one group of warps of its tiles walks.
struct GroupEntry {
    GroupItem item;
    int chain;
    double stage_us = kGroupStageUs + 2.0 * kGroupShiftUs;
};
inline void group_entry(const Shape& s, const Config& c, const void* A, const void* B, void* C, GroupEntry* e)
{
    e->chain = group_item(s, c, A, B, C, &e->item);
    const int64_t lda = s.layoutA == ADAPT_ROW_MAJOR ? s.K : s.M, ldb = s.layoutB == ADAPT_ROW_MAJOR ? s.N : s.K;
    e->stage_us = kGroupStageUs + ((((uintptr_t)A & 15) || lda % 8) ? kGroupShiftUs * std::min(1.0, (double)s.M / 64.0) : 0.0) +
                 ((((uintptr_t)B & 15) || ldb % 8) ? kGroupShiftUs * std::min(1.0, (double)s.N / 64.0) : 0.0);
}

// Tiles whose chain the launch would wait for are shared between two CTAs (four pieces) or four (eight, sixteen), whose groups of warps then walk
// one piece each, or two: log2 of the CTAs, and the chain that is left.
struct GroupShare { int log2, chain; };
inline GroupShare group_share(const GroupEntry& e, double average_us)
{
    const GroupItem& it = e.item;
    if (it.pieces < 4 || 2.0 * e.chain * e.stage_us <= average_us) return {0, e.chain};
    const int log2 = it.pieces == 4 ? 1 : 2, chain = it.pieces / (2 << log2) * (int)ceil_div(it.k_per_piece, kClusterKS);
    if ((e.chain - chain) * e.stage_us < 1.0) return {0, e.chain};
    return {log2, chain};
}

// The order of a list's entries in the launch.  The tile with the longest chain is what a short list waits for: its tiles are shared where the chain is
// longer than half of what a CTA slot (two per SM) has to do on average, where that takes off more than the exchange and the further CTAs
// cost, and the list stays within four CTAs per SM.  Beyond, the SMs are busy while the long chains run (the longest come first), and clusters, which
// start when four slots of a GPC are free, cost more than they save: 8 layers of 16 .. 1024 a side 9.7 -> 7.7 us, 24 layers 19.3 -> 11.8,
// 15 layers with K > 256 19.4 -> 17.5, but 47 layers (1018 CTAs shared, 762 not) 20.9 -> 27.3.  Of 344 lists in which sharing every
// long chain had been the rule, this one takes 1.003 of the better of both ways on average, that one 1.010 (8 layers of 200 x 200 x 512 beside 20 small
// ones: 9.1 us and 13.6).
inline void group_order(GroupEntry* e, size_t n, int n_sm)
{
    const double slots = 2.0 * n_sm;
    double work = 0.0, longest = 0.0, left = 0.0;
    int64_t tiles = 0, ctas = 0;
    for (size_t j = 0; j < n; ++j) {
        const double us = e[j].chain * e[j].stage_us;
        work += e[j].item.tiles * us;
        tiles += e[j].item.tiles;
        longest = std::max(longest, us);
    }
    GroupShare share[kGroupMax];
    for (size_t j = 0; j < n; ++j) {
        share[j] = group_share(e[j], work / slots);
        ctas += (int64_t)e[j].item.tiles << share[j].log2;
        left = std::max(left, share[j].chain * e[j].stage_us);
    }
    const double busy = (work + kGroupTileUs * tiles) / slots;         // what the slots have to do in any case
    const double saved = std::max(longest, busy) - std::max(left, busy);
    const double rounds = (std::max((double)ctas, slots) - std::max((double)tiles, slots)) / slots;
    if (ctas <= 4 * (int64_t)n_sm && saved > kGroupExchangeUs + kGroupRoundUs * rounds)
        for (size_t j = 0; j < n; ++j) {
            e[j].item.share_log2 = (short)share[j].log2;
            e[j].chain = share[j].chain;
        }
    // (by keys: sorting the entries themselves is a tenth of what the host spends on a list)
    uint32_t key[kGroupMax];
    for (size_t j = 0; j < n; ++j) key[j] = (uint32_t)(3 - e[j].item.share_log2) << 24 | (uint32_t)(0xffff - std::min(e[j].chain, 0xffff)) << 8 | (uint32_t)j;
    std::sort(key, key + n);
    GroupEntry as_given[kGroupMax];
    std::copy(e, e + n, as_given);
    for (size_t j = 0; j < n; ++j) e[j] = as_given[key[j] & 0xff];
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
