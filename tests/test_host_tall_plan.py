"""The schedule of the tall pair tiles, compiled on its own: every 256-row block of every column is computed once, whatever the number of
rows, columns and SM pairs, and the halves of a tile are blocks of one row class."""
from test_host_group_plan import build_and_run

PROGRAM = r"""
#include <cstdio>
#include <set>
#include <vector>
#include "adapt_internal.h"
using namespace adapt;

template <bool CLS>
int check(int64_t M, int P_n, int slots)
{
    double waves = 0;
    const TallWork w = tall_schedule(M, P_n, CLS, slots, &waves);
    const int64_t blocks = CLS ? (M + 2047) / 2048 * 8 : (M + 255) / 256;
    const int grid = std::min(w.big + w.halves, slots);
    std::vector<int> seen(blocks * P_n, 0);
    double longest = 0;
    int bad = 0;
    for (int slot = 0; slot < grid; ++slot) {
        TallItem t;
        double len = 0;
        for (int it = 0; tall_item<CLS>(w, slot, grid, it, t); ++it) {
            for (int h = 0; h < (t.two ? 2 : 1); ++h) {
                const int blk = h ? t.blk1 : t.blk0;
                if (blk < 0 || blk >= blocks || t.nb < 0 || t.nb >= P_n) { ++bad; continue; }
                ++seen[(int64_t)blk * P_n + t.nb];
            }
            if (t.two && CLS && (t.blk0 & 7) != (t.blk1 & 7)) ++bad;
            if (t.acc < 0 || t.acc > 1 || (t.two && t.acc)) ++bad;
            len += t.two ? 1.0 : 0.5;
        }
        longest = std::max(longest, len);
    }
    for (int s : seen) bad += s != 1;
    if (longest > waves + 0.5) ++bad;
    if (bad) printf("M %lld P_n %d slots %d classes %d: %d wrong, %.1f waves, longest slot %.1f\n", (long long)M, P_n, slots, (int)CLS, bad, waves, longest);
    return bad;
}

int main()
{
    int bad = 0;
    for (int slots : {74, 66, 5, 1})
        for (int P_n : {1, 2, 3, 7, 16, 56, 100})
            for (int64_t M : {1, 255, 256, 257, 512, 513, 768, 1000, 2048, 2049, 4096, 4097, 6144, 8192, 12288, 20001, 33000}) {
                bad += check<false>(M, P_n, slots);
                bad += check<true>(M, P_n, slots);
            }
    return bad != 0;
}
"""


def test_tall_tiles_cover_the_output_once(tmp_path):
    r = build_and_run(tmp_path, PROGRAM)
    assert r.returncode == 0, r.stdout + r.stderr
