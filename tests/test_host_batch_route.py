"""The host rules of strided batches, compiled on their own: how much the copies of unaligned operands hold at a time, and that the parts of
a batch cover its entries."""
from test_host_group_plan import build_and_run

PROGRAM = r"""
#include <cstdio>
#include <random>
#include "batch_route.h"
using namespace adapt;

int main()
{
    const Machine m;
    const Calib cal;
    std::mt19937_64 rng(3);
    auto upto = [&](int64_t hi) { return (int64_t)1 + (int64_t)(rng() % (unsigned long long)hi); };
    int tensor = 0, several = 0, grouped = 0, loops = 0, bad = 0;
    for (int trial = 0; trial < 1500; ++trial) {
        Shape s;
        s.M = upto(trial % 2 ? 200 : 3000); s.N = upto(trial % 3 ? 300 : 4000); s.K = upto(trial % 5 ? 500 : 6000);
        s.layoutA = (int)(rng() % 2); s.layoutB = (int)(rng() % 2);
        if (trial % 4 == 0) { s.M = round_up(s.M, 16); s.N = round_up(s.N, 16); s.K = round_up(s.K, 16); }
        const int64_t batch = 2 + upto(trial % 7 ? 60 : 5000), gap = trial % 9 ? 0 : upto(24);
        std::vector<Config> all;
        enumerate_configs(s, m, cal, &all);
        const bool a_rm = s.layoutA == ADAPT_ROW_MAJOR, b_rm = s.layoutB == ADAPT_ROW_MAJOR;
        const uintptr_t base = 4096 + (trial % 6 ? 0 : 2 * upto(8));
        const BatchOperand a((const void*)base, a_rm ? s.K : s.M, a_rm ? s.M : s.K, batch, s.M * s.K + gap);
        const BatchOperand b((const void*)base, b_rm ? s.N : s.K, b_rm ? s.K : s.N, batch, trial % 8 ? s.K * s.N + gap : 0);
        const BatchRoute r = batch_route(s, all[0], m, batch, all[0].family == ADAPT_FAM_CLUSTER, true, a, b, trial % 2 != 0);
        tensor += r.kind == kBatchUmma; grouped += r.kind == kBatchGroup; loops += r.kind == kBatchLoop;
        bool ok = r.kind == kBatchUmma || r.chunk == batch;
        if (r.kind == kBatchUmma) {
            several += r.chunk < batch;
            ok &= r.chunk >= 1 && r.chunk <= batch && a.ok && b.ok;
            int64_t first = 0;
            while (first < batch) {
                const int64_t n = std::min(r.chunk, batch - first);
                const BatchOperand x = a.part(first, n), y = b.part(first, n);
                ok &= (int64_t)(x.bytes() + y.bytes()) <= kBatchCopyBytes;
                ok &= (uintptr_t)x.src == base + (uintptr_t)(2 * first * a.stride) && x.entries == n;
                ok &= y.shared ? (uintptr_t)y.src == base && y.entries == 1 : (uintptr_t)y.src == base + (uintptr_t)(2 * first * b.stride) && y.entries == n;
                // a copy holds all rows of its entries at the padded pitch; what is read in place starts on a 16-byte boundary
                ok &= !x.copy || x.bytes() >= (size_t)(n * x.outer * x.pitch * 2);
                ok &= x.copy || ((uintptr_t)x.src % 16 == 0 && x.entry_stride * 2 % 16 == 0 && x.pitch == x.inner);
                first += n;
            }
        }
        if (!ok && bad++ < 10) printf("trial %d: %lld x %lld x %lld, %lld entries: kind %d, %lld at a time\n", trial, (long long)s.M, (long long)s.N, (long long)s.K, (long long)batch, r.kind, (long long)r.chunk);
    }
    printf("%d on the tensor-core kernel (%d in several launches), %d grouped, %d entry by entry\n", tensor, several, grouped, loops);
    return bad || tensor < 300 || several < 30 || grouped < 20;
}
"""


def test_copies_of_a_strided_batch_are_bounded(tmp_path):
    r = build_and_run(tmp_path, PROGRAM)
    assert r.returncode == 0, r.stdout + r.stderr
    print(r.stdout)
