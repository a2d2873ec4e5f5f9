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


@pytest.fixture
def tall_preferred():
    """The model made to take tall tiles wherever they are legal and compute-bound, whatever its constants."""
    adapt_build.build()
    ab.load()
    old = ab.adapt_get_calibration("eta_tall")
    ab.adapt_set_calibration("eta_tall", 3.0)
    yield
    ab.adapt_set_option("shuffle_k", 0)
    ab.adapt_set_calibration("eta_tall", old)


C, D, D_OFF = 1 << 20, 1 << 30, (1 << 30) + 8          # addresses, never followed


# (others: 4 splits, 7 splits, uncut tiles over a copy, in place, of row classes)
@pytest.mark.parametrize("M,N,K", [(1203, 4416, 8704), (413, 4736, 8960), (5366, 16320, 901), (8192, 4096, 1024), (8192, 2048, 4093)])
def test_second_configuration_is_the_best_on_other_tiles(tall_preferred, M, N, K):
    plan = ab.adapt_matmul_plan(M, N, K, ab.BF16)
    key = ab.adapt_plan_info(plan).tiling_key
    assert ab.adapt_plan_info(plan).BM == 512
    other = next(c for c in ab.adapt_plan_candidates(M, N, K, ab.BF16) if c.BM != 512)
    first, second = {(C, 0, False), (C, D, True), (C + 32, D + 16, True)}, {(C + 16, 0, False), (C + 2, D, True), (C, D_OFF, True), (C, D_OFF, False)}
    (first if K >= 1024 else second).add((C, D, False))
    for call in first:
        assert ab.adapt_plan_info_call(plan, *call).tiling_key == key, call
    for call in second:
        assert ab.adapt_plan_info_call(plan, *call).tiling_key == other.tiling_key, call
    ab.adapt_set_option("shuffle_k", 1)                 # (row classes have no such order)
    assert ab.adapt_plan_info_call(plan, C).tiling_key == (key if ab.adapt_plan_info(plan).srcA == 3 else other.tiling_key)


def test_second_configuration_of_a_forced_key_keeps_its_tiles_and_sources(tall_preferred):
    for M, N, K, lA, lB in [(1203, 4416, 8704, 0, 0), (300, 272, 80, 1, 1), (4501, 688, 333, 0, 0), (1001, 688, 333, 0, 0)]:
        tall = next(c for c in ab.adapt_plan_candidates(M, N, K, ab.F16, lA, lB) if c.BM == 512)
        plan = ab.adapt_matmul_plan_forced(M, N, K, ab.F16, lA, lB, tall.tiling_key)
        assert ab.adapt_plan_info_call(plan, C).tiling_key == tall.tiling_key
        i = ab.adapt_plan_info_call(plan, C + 2)
        assert (i.family, i.BM, i.BN, i.P_k, i.srcA, i.srcB, i.fused, i.streamk) == (ab.FAM_UMMA_2CTA, 256, 256, 1, tall.srcA, tall.srcB, 0, 0)
        assert any(c.tiling_key == i.tiling_key for c in ab.adapt_plan_candidates(M, N, K, ab.F16, lA, lB))


def test_second_configuration_of_a_loaded_plan(tall_preferred, tmp_path):
    M, N, K = 1205, 4416, 8704
    cands = ab.adapt_plan_candidates(M, N, K, ab.BF16)
    assert cands[0].BM == 512
    path = tmp_path / "table.txt"
    ab.adapt_matmul_plan(M, N, K, ab.BF16)
    ab.adapt_plan_table_save(str(path))
    line = [x for x in path.read_text().splitlines() if f"{M} {N} {K}" in x.replace(",", " ")]
    assert len(line) == 1
    path.write_text("\n".join([path.read_text().splitlines()[0]] + [line[0].replace(str(M), str(M + 1), 1)]) + "\n")
    assert ab.adapt_plan_table_load(str(path)) == 1
    plan = ab.adapt_matmul_plan(M + 1, N, K, ab.BF16)
    other = next(c for c in ab.adapt_plan_candidates(M + 1, N, K, ab.BF16) if c.BM != 512)
    assert ab.adapt_plan_info(plan).BM == 512 and ab.adapt_plan_info_call(plan, C + 4).tiling_key == other.tiling_key
