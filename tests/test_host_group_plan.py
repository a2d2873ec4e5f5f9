"""The host rules of grouped launches, compiled on their own: every configuration that a plan table may name gets a kernel whose
shared memory and division of the k range hold it."""
import os
import subprocess

ROOT = os.path.dirname(os.path.dirname(os.path.abspath(__file__)))
CSRC = os.path.join(ROOT, "paper_2608_10803_b200", "csrc")

PROGRAM = r"""
#include <cstdio>
#include "group_plan.h"
using namespace adapt;

static int bad = 0;
static void check(bool ok, const char* what, const Shape& s, const Config& c)
{
    if (ok) return;
    if (bad++ < 10) printf("%s: %lld x %lld x %lld family %d pieces %d\n", what, (long long)s.M, (long long)s.N, (long long)s.K, c.family, c.cluster);
}

int main()
{
    const Machine m;
    const Calib cal;
    int grouped = 0, several = 0;
    for (int64_t mn : {1, 64, 65, 128})
        for (int64_t K = 1; K <= 200; ++K) {
            Shape s;
            s.M = s.N = mn; s.K = K;
            std::vector<Config> all;
            enumerate_configs(s, m, cal, &all);
            for (const Config& c : all) {
                if (!group_eligible(s, c)) continue;
                Config again;
                check(config_from_key(s, pack_tiling_key(s, c), m, cal, &again), "a candidate's key is refused", s, c);
                ++grouped;
                several += c.family == ADAPT_FAM_CLUSTER && c.cluster > 1 && K <= kClusterKS;
                GroupItem it;
                const int chain = group_item(s, c, nullptr, nullptr, nullptr, &it);
                GroupParams p;
                group_clear(p);
                group_add(p, it, chain);
                group_add(p, it, chain);
                check(p.item[0].tile_end == it.tiles && p.item[1].tile_end == 2 * it.tiles, "tiles", s, c);
                const GroupForm f = group_form(p);
                // one stage, one CTA per tile: the k range is one piece of one stage
                check(!f.short_k || it.pieces == 0 || (it.pieces == 1 && K <= kClusterKS), "short kernel for several pieces or stages", s, c);
                check(f.short_k ? f.smem_bytes >= kClusterStageBytes : f.smem_bytes >= 2 * p.ring * kClusterStageBytes, "shared memory", s, c);
                // a ring of one stage is never refilled
                check(p.ring > 1 || chain <= 1, "ring", s, c);
                // the pieces cover the k range, none of them empty
                check(it.pieces == 0 || ((int64_t)it.pieces * it.k_per_piece >= K && (int64_t)(it.pieces - 1) * it.k_per_piece < K), "pieces", s, c);
            }
        }
    printf("%d configurations, %d of several pieces within one stage\n", grouped, several);
    return bad || grouped < 500 || several < 20;
}
"""


def build_and_run(tmp_path, program):
    src, exe = tmp_path / "check.cpp", tmp_path / "check"
    src.write_text(program)
    subprocess.run(["g++", "-std=c++17", "-O1", "-I", CSRC, "-I", os.path.join(ROOT, "include"), "-o", str(exe), str(src),
                    os.path.join(CSRC, "adapt_select.cpp")], check=True)
    return subprocess.run([str(exe)], capture_output=True, text=True, timeout=120)


def test_every_groupable_configuration_gets_a_kernel_that_holds_it(tmp_path):
    r = build_and_run(tmp_path, PROGRAM)
    assert r.returncode == 0, r.stdout + r.stderr


def test_clusters_that_all_fit_get_an_sm_per_cta(tmp_path):
    """Shared memory of a cluster launch: more than half of an SM's where all clusters run at once with an SM per CTA, never less than
    the ring, never more than a CTA may have."""
    r = build_and_run(tmp_path, r"""
#include <cstdio>
#include "adapt_internal.h"
using namespace adapt;
int main()
{
    const Machine m;
    int alone = 0, shared = 0;
    for (int cs : {1, 2, 4, 8, 16})
        for (int64_t tiles = 1; tiles * cs <= 2 * m.n_sm; ++tiles)
            for (int ring = 1; ring <= kClusterMaxRing; ++ring) {
                const int bytes = cluster_launch_bytes(ring, cs, tiles, m.n_sm);
                const bool fits = cs > 1 && tiles <= cluster_slots(cs, m.n_sm);
                if (bytes < cluster_smem_bytes(ring) || bytes > m.smem_bytes || (2 * (bytes + 1024) > 228 * 1024) != fits) return 1;
                alone += fits;
                shared += !fits;
            }
    return alone == 0 || shared == 0;
}
""")
    assert r.returncode == 0, r.stdout + r.stderr
