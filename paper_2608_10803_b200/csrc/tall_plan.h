// How a shape is cut into tall pair tiles (tall_gemm.cuh) and who computes which: plain C++, shared by the model, the launcher and the kernel.
#pragma once

#include <cstdint>

#ifdef __CUDACC__
#define ADAPT_HOST_DEVICE __host__ __device__ __forceinline__
#else
#define ADAPT_HOST_DEVICE inline
#endif

namespace adapt {

constexpr int kTallGroup = 8;            // rasterisation: rows of tiles per group, 4096 rows of A as for the 256-row tiles

// A tile is two 256-row blocks.  Rows of C are blocks of 256 consecutive ones, or, with the 8 row classes of an unaligned A, block 8 g + j
// is the rows 2048 g + j + 8 i; the two blocks of a tile are of one class.
struct TallWork {
    int P_n;                             // columns of tiles
    int row_pairs, odd_rows;             // rows of whole tiles; rows of blocks without a partner (the last one of an odd number, per class)
    int big;                             // tiles computed as such; the rest as their 256-row halves,
    int split;                           // this many,
    int halves;                          // ... and these with the blocks of the odd rows
    int last, free_slots;                // slots with a whole tile in the last wave, and without (none: 0, 0)
};

// The length of a schedule whose whole tiles take t_tile and whose single blocks take t_half: whole waves, then the blocks, first on the slots
// without a tile in the last wave (two in a tile's time).
inline double tall_length(const TallWork& w, int64_t slots, double t_tile, double t_half)
{
    const int64_t last = w.big % slots, room = last ? 2 * (slots - last) : 0, more = w.halves > room ? w.halves - room : 0;
    const bool twos = last && 2 * w.halves > room;                   // some slot has two blocks in the last wave's time
    return (double)(w.big / slots) * t_tile + (last ? (twos && 2.0 * t_half > t_tile ? 2.0 * t_half : t_tile) : 0.0) + (double)((more + slots - 1) / slots) * t_half;
}

// The tiles that do not fill a whole wave of slots (SM pairs) are cut when all the halves then fit one wave of half the length: they
// bring B twice, but 2048 x 14336 x 4096, 224 tiles on 74 pairs, takes 3.5 waves instead of 4.
// *waves: the length of the schedule in whole tiles.
inline TallWork tall_schedule(int64_t M, int64_t P_n, bool classes, int64_t slots, double* waves = nullptr)
{
    const int64_t n = classes ? 8 : 1, blocks = (M + 256 * n - 1) / (256 * n);          // blocks of 256 rows (of one class)
    const int64_t pairs = blocks / 2 * n, odd = blocks % 2 * n;
    const int64_t tiles = pairs * P_n, rest = tiles % slots, single = odd * P_n;
    const bool cut = rest > 0 && 2 * rest + single <= slots;
    TallWork w;
    w.P_n = (int)P_n;
    w.row_pairs = (int)pairs;
    w.odd_rows = (int)odd;
    w.big = (int)(cut ? tiles - rest : tiles);
    w.split = (int)(cut ? 2 * rest : 0);
    w.halves = (int)(w.split + single);
    const int64_t n_slots = w.big + w.halves < slots ? w.big + w.halves : slots;
    w.last = n_slots ? (int)(w.big % n_slots) : 0;
    w.free_slots = w.last ? (int)(n_slots - w.last) : 0;
    if (waves) *waves = tall_length(w, slots, 1.0, 0.5);
    return w;
}

// A unit of work: a whole tile (two), or one of its blocks, on accumulator `acc`.
struct TallItem {
    int blk0, blk1, nb;                  // blocks of the upper and the lower half, column of tiles
    int acc;
    bool two;
};

// The it-th item of a slot: its whole tiles, then its share of the single blocks.  (A single block behind the whole tile of a slot, where
// another slot had none: 1771 x 4736 x 6288, 57 tiles and 19 single blocks on 74 pairs, with zero operands 100 us, 77 this way.)
template <bool CLS>
ADAPT_HOST_DEVICE bool tall_item(const TallWork& p, int slot, int n_slots, int it, TallItem& w)
{
    const int mine = slot < p.big ? (p.big - slot - 1) / n_slots + 1 : 0;
    int t, h = 0;
    w.acc = 0;
    w.two = it < mine;
    if (w.two) {
        t = slot + it * n_slots;
    } else {
        // two for each slot without a tile in the last wave (which the others spend on a whole tile), then one for every slot in turn
        const int first = slot < p.last ? slot + p.free_slots : slot - p.last;
        int j = it - mine;
        w.acc = j & 1;
        if (p.last && slot >= p.last) {
            h = first + j * p.free_slots;
            j -= 2;
        }
        if (j >= 0) h = 2 * p.free_slots + first + j * n_slots;
        if (h >= p.halves) return false;
        t = p.big + (h >> 1);
        if (h >= p.split) {                                    // the odd rows
            const int o = h - p.split;
            w.nb = o / p.odd_rows;
            w.blk0 = w.blk1 = 2 * p.row_pairs + (o - w.nb * p.odd_rows);
            return true;
        }
    }
    const int group_size = kTallGroup * p.P_n;
    const int g = t / group_size, first_m = g * kTallGroup;
    const int gm = p.row_pairs - first_m < kTallGroup ? p.row_pairs - first_m : kTallGroup;
    const int r = t - g * group_size;
    const int mp = first_m + r % gm;
    w.nb = r / gm;
    w.blk0 = CLS ? (mp >> 3) * 16 + (mp & 7) : 2 * mp;
    w.blk1 = w.blk0 + (CLS ? 8 : 1);
    if (!w.two) w.blk0 = w.blk1 = (h & 1) ? w.blk1 : w.blk0;
    return true;
}

}  // namespace adapt
