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


SHARED = r"""
#include <cstdio>
#include <map>
#include <random>
#include <vector>
#include "group_plan.h"
using namespace adapt;

int main()
{
    std::mt19937 rng(7);
    int bad = 0, shared_lists = 0, fillers = 0;
    for (int trial = 0; trial < 3000; ++trial) {
        const int n = 1 + rng() % (trial % 3 ? 6 : 64);
        std::vector<GroupEntry> e(n);
        for (GroupEntry& x : e) {
            const int pieces[] = {0, 1, 1, 2, 4, 4, 8, 16};
            x.item = GroupItem();
            x.item.pieces = (short)pieces[rng() % 8];
            x.item.k_per_piece = x.item.pieces ? 16 * (1 + rng() % 12) : 0;
            x.item.tiles = 1 + rng() % 30;
            x.item.K = x.item.pieces * x.item.k_per_piece;
            const int spp = (x.item.k_per_piece + 63) / 64;
            x.chain = x.item.pieces <= 1 ? 1 + rng() % 3 : x.item.pieces / 2 * spp;
            x.item.M = x.chain;                                     // (kept to compare with)
        }
        group_order(e.data(), n, 148);
        int64_t ctas = 0, shared = 0;
        for (const GroupEntry& x : e) {
            const int share = 1 << x.item.share_log2;
            ctas += x.item.tiles * share;
            shared += share > 1;
            // no more than two pieces for a group of warps of a shared tile, and the chain that is left holds them
            if (share > 1 ? x.item.pieces > 4 * share || x.item.pieces < 2 * share || x.chain >= x.item.M || x.chain < x.item.pieces / (2 * share) : x.chain != x.item.M) ++bad;
        }
        if (shared && ctas > 4 * 148) ++bad;
        GroupParams p;
        group_clear(p);
        for (GroupEntry& x : e) group_add(p, x.item, x.chain);
        const int grid = group_grid(p);
        shared_lists += p.sync_ctas > 0;
        if (p.sync_ctas % kGroupCluster || (p.sync_ctas && grid % kGroupCluster)) ++bad;
        std::map<std::pair<int, int>, std::vector<int>> who;       // (item, tile) -> CTAs in order of q
        for (int cta = 0; cta < grid; ++cta) {
            GroupPlace w;
            if (!group_place(p, cta, w)) { ++fillers; continue; }
            std::vector<int>& v = who[{w.item, w.tile}];
            if ((int)v.size() != w.q || w.entry != 0 || w.tile >= p.item[w.item].tiles) ++bad;
            v.push_back(cta);
            // the CTAs of a shared tile wait at two cluster barriers, and so do all of their cluster; no others do
            if ((p.item[w.item].share_log2 > 0) != (cta < p.sync_ctas)) ++bad;
        }
        int tiles = 0;
        for (int i = 0; i < p.count; ++i) tiles += p.item[i].tiles;
        if ((int)who.size() != tiles) ++bad;
        for (auto& kv : who) {
            const int share = 1 << p.item[kv.first.first].share_log2;
            if ((int)kv.second.size() != share || kv.second.back() - kv.second[0] != share - 1) ++bad;
            if (share > 1 && kv.second[0] / kGroupCluster != kv.second.back() / kGroupCluster) ++bad;
            // buffers of the pieces' sums: two per piece of a group of warps, inside the rings
            if (share > 1 && p.item[kv.first.first].pieces / share * kClusterStageBytes > group_form(p).smem_bytes) ++bad;
        }
        if (group_form(p).short_k && p.sync_ctas) ++bad;
    }
    printf("%d lists with shared tiles, %d CTAs without work, %d wrong\n", shared_lists, fillers, bad);
    return bad || shared_lists < 500 || fillers < 100;
}
"""


def test_shared_tiles_get_their_ctas_in_one_cluster(tmp_path):
    r = build_and_run(tmp_path, SHARED)
    assert r.returncode == 0, r.stdout + r.stderr


WORTH = r"""
#include <cmath>
#include <cstdio>
#include <vector>
#include "group_plan.h"
using namespace adapt;

struct Dims { int64_t M, N, K; };
// The entries of a list as the library plans them, in launch order; bit s: some tile is shared by 2^s CTAs.
static int shares(const std::vector<Dims>& list, uintptr_t offset = 0)
{
    std::vector<GroupEntry> e;
    for (const Dims& d : list) {
        Shape s;
        s.M = d.M; s.N = d.N; s.K = d.K;
        std::vector<Config> all;
        enumerate_configs(s, Machine(), default_calib(), &all);
        if (!group_eligible(s, all[0])) { printf("%lld x %lld x %lld is not for the grouped launch\n", (long long)d.M, (long long)d.N, (long long)d.K); return -1; }
        e.emplace_back();
        group_entry(s, all[0], (const void*)(4096 + offset), (const void*)8192, (void*)16384, &e.back());
    }
    group_order(e.data(), e.size(), 148);
    int bits = 0;
    for (const GroupEntry& x : e) bits |= 1 << x.item.share_log2;
    return bits;
}
static int bad = 0;
static void check(bool ok, const char* what) { if (!ok) { printf("%s\n", what); ++bad; } }

int main()
{
    // the lists of the bit-for-bit test on the GPU: tiles of one, two and four CTAs
    const std::vector<std::vector<Dims>> lists = {{{84, 39, 1014}, {20, 30, 40}}, {{504, 209, 576}, {100, 100, 100}, {30, 7, 20}},
        {{64, 64, 1024}, {65, 63, 1000}, {17, 763, 618}, {105, 845, 611}, {1, 1, 500}}, {{38, 48, 787}, {48, 38, 808}, {1, 70, 790}},
        {{64, 128, 1008}, {16, 200, 520}, {129, 1, 400}, {300, 200, 50}, {10, 10, 65}, {33, 65, 130}, {7, 9, 11}, {40, 342, 267}}};
    int seen = 0;
    for (const auto& l : lists) seen |= shares(l);
    check(seen == 7, "tiles of one, two and four CTAs");
    // eight layers of 16 tiles beside 20 small ones: not where four CTAs to a tile are a round more
    auto beside = [&](int count, Dims d) { std::vector<Dims> l(20, Dims{40, 40, 40}); l.insert(l.end(), count, d); return l; };
    for (int64_t K : {384, 500, 512}) check(shares(beside(8, {200, 200, K})) == 1, "many tiles of medium chains");
    check(shares(beside(1, {128, 65, 500})) == (1 | 4) && shares(beside(4, {64, 64, 1024})) == (1 | 4), "long chains of a few tiles");
    // a stage takes longer by the shift of each operand off 16-byte boundaries: its rows, its buffer, as many rows as a tile has of it
    auto stage = [&](Dims d, uintptr_t a, uintptr_t b) {
        Shape s;
        s.M = d.M; s.N = d.N; s.K = d.K;
        std::vector<Config> all;
        enumerate_configs(s, Machine(), default_calib(), &all);
        GroupEntry e;
        group_entry(s, all[0], (const void*)a, (const void*)b, nullptr, &e);
        return e.stage_us;
    };
    check(stage({64, 64, 512}, 4096, 8192) == kGroupStageUs && stage({64, 64, 512}, 4098, 8192) == kGroupStageUs + kGroupShiftUs, "a buffer");
    check(std::abs(stage({64, 63, 511}, 4096, 8192) - (kGroupStageUs + kGroupShiftUs * (1.0 + 63.0 / 64.0))) < 1e-12 && stage({16, 64, 511}, 4096, 8192) == kGroupStageUs + kGroupShiftUs / 4, "rows");
    check(shares(std::vector<Dims>(60, Dims{130, 65, 389})) == 1, "busy SMs");
    return bad;
}
"""


def test_tiles_are_shared_where_it_pays(tmp_path):
    r = build_and_run(tmp_path, WORTH)
    assert r.returncode == 0, r.stdout + r.stderr
