"""The tables of timed configurations that the calibration tool reads: every configuration keeps its own line and its own group."""
import pytest

from paper_2608_10803_b200 import binding as ab
from paper_2608_10803_b200 import build as adapt_build
from paper_2608_10803_b200 import calibrate

from test_host_group_plan import build_and_run


@pytest.fixture(scope="module", autouse=True)
def lib():
    adapt_build.build()
    return ab.load()


def test_table_of_timed_configurations_tells_both_pair_tiles_apart(tmp_path):
    """256 x 256 and 512 x 256 pair tiles of the same depth, split and sources are two lines of a table: each keeps its own time."""
    shape = (8192, 8192, 8192, 1)
    pair = {c.BM: c for c in ab.adapt_plan_candidates(*shape) if c.family == ab.FAM_UMMA_2CTA and c.BN == 256 and c.stages == 4 and c.P_k == 1 and not c.streamk}
    assert set(pair) == {256, 512}
    path = tmp_path / "cand.csv"
    path.write_text("".join(",".join(r) + "\n" for r in [calibrate.COLUMNS] + [calibrate.table_row(shape, c, 700.0 + bm) for bm, c in pair.items()]))
    timed = calibrate.TimedSet([str(path)])
    assert sorted(timed.shapes[shape].values()) == [956.0, 1212.0]
    assert timed.metrics(ab)["mean"] == (1212.0 / 956.0 if pair[512].predicted_us < pair[256].predicted_us else 1.0)
    rows = [dict(zip(calibrate.COLUMNS, calibrate.table_row(shape, pair[bm], 1.0))) for bm in (256, 512)]
    assert [calibrate.group_of(r) for r in rows] == [20, 36]


GROUPS_PROGRAM = r"""
#include <cstdio>
#include "adapt_internal.h"
using namespace adapt;
int main()
{
    const char* family[] = {"umma_1cta", "umma_2cta", "skinny", "simt", "cluster"};
    Machine m;
    m.family_mask = 0x1F;
    for (int64_t M : {8, 300, 4500}) for (int64_t N : {8, 272, 331, 1024}) for (int64_t K : {64, 333, 4096}) for (int lb : {0, 1}) {
        Shape s;
        s.M = M; s.N = N; s.K = K; s.layoutB = lb;
        std::vector<Config> all;
        enumerate_configs(s, m, default_calib(), &all);
        for (const Config& c : all)
            printf("%s,%d,%d,%d,%d,%d,%d,%d,%d,%d\n", family[c.family], c.BM, c.BN, c.P_k, c.cluster, c.fused, c.streamk, c.srcA, c.srcB, calib_group(c));
    }
}
"""


def test_calibration_groups_of_the_tool_are_the_selectors(tmp_path):
    seen = set()
    r = build_and_run(tmp_path, GROUPS_PROGRAM)
    assert r.returncode == 0, r.stdout + r.stderr
    for line in r.stdout.splitlines():
        *values, group = line.split(",")
        row = dict(zip("family,BM,BN,P_k,cluster,fused,streamk,srcA,srcB".split(","), values))
        assert calibrate.group_of(row) == int(group), line
        seen.add(int(group))
    assert {20, 22, 36, 37, 38} <= seen
