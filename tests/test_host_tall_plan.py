"""The schedule of the tall pair tiles, compiled on its own: every 256-row block of every column is computed once, whatever the number of
rows, columns and SM pairs, and the halves of a tile are blocks of one row class."""
import pytest

from paper_2608_10803_b200 import binding as ab
from paper_2608_10803_b200 import build as adapt_build

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


BALANCE = r"""
#include <cstdio>
#include "adapt_internal.h"
using namespace adapt;

template <bool CLS>
int check(int64_t M, int P_n, int slots)
{
    double waves = 0, longest = 0;
    const TallWork w = tall_schedule(M, P_n, CLS, slots, &waves);
    const int grid = std::min(w.big + w.halves, slots);
    for (int slot = 0; slot < grid; ++slot) {
        TallItem t;
        double len = 0;
        for (int it = 0; tall_item<CLS>(w, slot, grid, it, t); ++it) len += t.two ? 1.0 : 0.5;
        longest = std::max(longest, len);
    }
    if (longest == waves) return 0;
    printf("M %lld P_n %d slots %d classes %d: %.1f waves, longest slot %.1f\n", (long long)M, P_n, slots, (int)CLS, waves, longest);
    return 1;
}

int main()
{
    int bad = 0;
    for (int slots : {74, 66, 5, 1})
        for (int P_n = 1; P_n <= 100; ++P_n)
            for (int64_t M = 300; M < 20000; M += 419) bad += check<false>(M, P_n, slots) + check<true>(M, P_n, slots);
    return bad != 0;
}
"""


def test_longest_slot_is_what_the_model_counts(tmp_path):
    r = build_and_run(tmp_path, BALANCE)
    assert r.returncode == 0, r.stdout[-2000:] + r.stderr


C, D, D_OFF = 1 << 20, 1 << 30, (1 << 30) + 8          # addresses, never followed


@pytest.fixture(autouse=True)
def library():
    adapt_build.build()
    ab.load()
    yield
    ab.adapt_set_option("shuffle_k", 0)


# in place, a short k range, over copies, of row classes; plans of the model's choice, and by their keys
@pytest.mark.parametrize("M,N,K,lA,lB", [(8192, 8192, 8192, 0, 0), (5366, 16320, 896, 0, 0), (8193, 4096, 2048, 1, 1), (5366, 16320, 2901, 0, 0), (12288, 688, 16991, 0, 0), (300, 272, 80, 1, 1)])
def test_calls_that_tall_tiles_cannot_serve_run_256_row_tiles_over_the_same_sources(M, N, K, lA, lB):
    cands = ab.adapt_plan_candidates(M, N, K, ab.BF16, lA, lB)
    tall = next(c for c in cands if c.BM == 512)
    plans = [ab.adapt_matmul_plan_forced(M, N, K, ab.BF16, lA, lB, tall.tiling_key)]
    if cands[0].BM == 512:
        plans.append(ab.adapt_matmul_plan(M, N, K, ab.BF16, lA, lB))
    assert len(plans) == 1 + (M > 300)
    served, others = {(C, 0, False), (C, D, True), (C + 32, D + 16, True)}, {(C + 16, 0, False), (C + 2, D, True), (C, D_OFF, True), (C, D_OFF, False)}
    (served if K >= 1024 else others).add((C, D, False))
    def runs_short(plan, call):
        i = ab.adapt_plan_info_call(plan, *call)
        assert any(c.tiling_key == i.tiling_key for c in cands)
        return (i.family, i.BM, i.BN, i.P_k, i.srcA, i.srcB, i.fused, i.streamk) == (ab.FAM_UMMA_2CTA, 256, 256, 1, tall.srcA, tall.srcB, 0, 0)

    for plan in plans:
        for call in served:
            assert ab.adapt_plan_info_call(plan, *call).tiling_key == tall.tiling_key, call
        for call in others:
            assert runs_short(plan, call), call
        ab.adapt_set_option("shuffle_k", 1)             # (row classes have no such order)
        assert runs_short(plan, (C, 0, False)) == (tall.srcA != 3)
        ab.adapt_set_option("shuffle_k", 0)


@pytest.mark.parametrize("M,N,K", [(16384, 16384, 4096), (40000, 16384, 4096), (8192, 8192, 8192), (6000, 14336, 4096)])
def test_both_pair_tiles_are_charged_the_same_readings_of_b(M, N, K):
    """Eight rows of tall tiles to a raster group are as many rows of A as sixteen of 256."""
    pair = {c.BM: c for c in ab.adapt_plan_candidates(M, N, K, ab.BF16) if c.family == ab.FAM_UMMA_2CTA and c.BN == 256 and c.P_k == 1 and not c.streamk}
    assert pair[512].hbm_bytes == pair[256].hbm_bytes


@pytest.mark.parametrize("M,N,K,lB", [(6668, 2112, 13504, 1), (5889, 2496, 9408, 0), (966, 10048, 16000, 0), (958, 15424, 12928, 0)])
def test_stream_k_is_not_given_up_for_a_mostly_idle_wave_of_tall_tiles(M, N, K, lB):
    cands = ab.adapt_plan_candidates(M, N, K, ab.F16, 0, lB)
    assert cands[0].streamk and [c.predicted_us for c in cands] == sorted(c.predicted_us for c in cands)
