"""Host-side logic of the C-ABI library, no GPU: exports, taxonomy, model closed forms,
candidate legality, plan cache.  The library's classifier and formulas are compared with the
oracle's (``oracle/taxonomy.py``), which is pinned to the paper separately."""
import ctypes
import os
import re
import time

import pytest

from oracle import taxonomy as tx
from paper_2608_10803_b200 import binding as ab
from paper_2608_10803_b200 import build as adapt_build
from paper_2608_10803_b200 import synth

ROOT = os.path.dirname(os.path.dirname(os.path.abspath(__file__)))
CLASS_ID = {tx.COMMON: 0, tx.SINGLE_CORE_SPLIT_K: 1, tx.MULTI_CORE_SPLIT_K: 2, tx.HYBRID_SPLIT_K: 3}


@pytest.fixture(scope="module", autouse=True)
def lib():
    adapt_build.build()
    return ab.load()


def test_library_exports_every_declared_symbol(lib):
    header = open(os.path.join(ROOT, "include", "adapt_matmul.h")).read()
    header = re.sub(r"/\*.*?\*/", "", header, flags=re.S)
    declared = set(re.findall(r"\b(adapt_[a-z_0-9]+)\s*\(", header))
    assert declared, "no declarations found"
    assert declared == set(ab.EXPORTS)
    for name in declared:
        assert hasattr(lib, name), name


def test_compute_without_device_fails_loudly(lib):
    import torch
    if torch.cuda.is_available():
        pytest.skip("device present")
    h = ab.adapt_matmul_plan(64, 64, 64, ab.F16)
    with pytest.raises(ab.AdaptError) as e:
        ab.adapt_matmul(h, 16, 16, 16, 0)
    assert e.value.status == ab.ERR_NOT_INIT


def worked_cases():
    out = []
    with open(os.path.join(ROOT, "tests", "golden", "taxonomy_cases.txt")) as f:
        for line in f:
            if line.startswith("#") or not line.strip():
                continue
            p = line.split()
            out.append(tuple(int(x) for x in p[:12]) + (p[12],))
    return out


@pytest.mark.parametrize("case", worked_cases())
def test_classifier_reproduces_worked_cases(case):
    _, M, N, K, m, n, m1, n1, N_core, S, _, _, template = case
    assert ab.adapt_classify(M, N, m, n, m1, n1, N_core, S) == CLASS_ID[template]


def test_classifier_matches_oracle_on_a_grid():
    for M in (1, 100, 1000, 5000, 100000):
        for N in (1, 64, 777, 4096):
            for (m, n) in ((128, 64), (128, 256), (256, 256)):
                for (nc, acc) in ((16, 128 << 10), (148, 128 << 10), (74, 256 << 10)):
                    want = CLASS_ID[tx.classify(M, N, m, n, m, n, nc, acc)]
                    assert ab.adapt_classify(M, N, m, n, m, n, nc, acc) == want
    assert ab.adapt_classify(0, 1, 1, 1, 1, 1, 1, 1) == -1


def test_volume_formulas_match_oracle():
    M, N, K = 12288, 688, 16991
    for (m1, n1) in ((128, 256), (256, 256), (128, 64)):
        assert ab.adapt_model_read_volume(M, N, K, m1, n1) == pytest.approx(float(tx.read_volume(M, N, K, m1, n1)), rel=1e-14)
    assert ab.adapt_model_write_volume(0, M, N, K, K, 64) == tx.write_volume_common(M, N)
    assert ab.adapt_model_write_volume(1, M, N, K, K, 512) == tx.write_volume_single_core_split_k(M, N, K, 512)
    assert ab.adapt_model_write_volume(2, M, N, K, 1024, 64) == tx.write_volume_multi_core_split_k(M, N, K, 1024)
    assert ab.adapt_model_write_volume(3, M, N, K, 1000, 300) == tx.write_volume_hybrid_split_k(M, N, K, 1000, 300)


def test_pipeline_formulas_match_oracle():
    for (Q, L, tM, tP, D) in ((1, 1, 3.0, 5.0, 1.0), (4, 9, 2.5, 1.5, 0.25), (7, 64, 1.0, 1.0, 3.0)):
        assert ab.adapt_model_pipeline(0, Q, L, tM, tP, D) == pytest.approx(Q * tx.t_baseline(L, tM, tP, D))
        assert ab.adapt_model_pipeline(1, Q, L, tM, tP, D) == pytest.approx(Q * tx.t_double_buffer(L, tM, tP, D))
        assert ab.adapt_model_pipeline(2, Q, L, tM, tP, D) == pytest.approx(tx.t_preload(Q, L, tM, tP, D))


def test_plan_is_cached_and_pointer_equal():
    a = ab.adapt_matmul_plan(1000, 1024, 1024, ab.F16)
    b = ab.adapt_matmul_plan(1000, 1024, 1024, ab.F16)
    c = ab.adapt_matmul_plan(1000, 1024, 1024, ab.BF16)
    d = ab.adapt_matmul_plan(1000, 1024, 1024, ab.F16, ab.COL_MAJOR, ab.ROW_MAJOR)
    assert a == b and a != c and a != d
    big = ab.adapt_matmul_plan(2_000_000, 8, 8, ab.F16)          # beyond the packed-key range
    assert big == ab.adapt_matmul_plan(2_000_000, 8, 8, ab.F16)


def test_plan_rejects_bad_arguments():
    with pytest.raises(ab.AdaptError) as e:
        ab.adapt_matmul_plan(-1, 4, 4, ab.F16)
    assert e.value.status == ab.ERR_INVALID_ARG
    with pytest.raises(ab.AdaptError) as e:
        ab.adapt_matmul_plan(1 << 31, 4, 4, ab.F16)
    assert e.value.status == ab.ERR_UNSUPPORTED
    with pytest.raises(ab.AdaptError):
        ab.adapt_matmul_plan(4, 4, 4, 7)


def test_every_shape_has_a_legal_candidate_and_info_is_consistent():
    shapes = [(1, 1, 1), (1, 4096, 4096), (7, 1024, 1024), (8192, 8192, 8192), (256, 256, 262144),
              (178, 71, 43035), (3067, 2, 75528), (6392, 8517, 4), (100000, 1024, 1024), (3, 256, 87087),
              (12288, 688, 16991), (17, 17, 17), (99999, 3, 5)]
    for (M, N, K) in shapes:
        for dt in (ab.F16, ab.BF16):
            cands = ab.adapt_plan_candidates(M, N, K, dt)
            assert cands, (M, N, K)
            assert all(cands[i].predicted_us <= cands[i + 1].predicted_us for i in range(len(cands) - 1))
            info = ab.adapt_plan_info(ab.adapt_matmul_plan(M, N, K, dt))
            assert (info.M, info.N, info.K, info.dtype) == (M, N, K, dt)
            assert info.flops == 2.0 * M * N * K
            assert info.P_k >= 1 and info.grid >= 1 and info.predicted_us > 0
            for c in cands:
                # capacity limits of Eq. 6
                if c.family in (ab.FAM_UMMA_1CTA, ab.FAM_UMMA_2CTA):
                    bn_cta = c.BN // c.cluster
                    # a stage holds the rows of A one box brings (128, or fewer for a short A) and BN columns of B
                    halo = c.BN % 64 != 0        # class tiles that own 32-byte units of C's shifted rows
                    # as few row classes as keep the rows of a class at one offset from a 32-byte boundary in C (and from a
                    # 16-byte one in an A read in place): 16 for an odd N, fewer for an even one
                    if halo:
                        for_c = next(n for n in (2, 4, 8, 16) if (n * N) % 16 == 0)
                        a_copied = K < 64 and not (K % 8 == 0 and K % 16 == 0)
                        for_a = 1 if a_copied else next(n for n in (1, 2, 4, 8) if (n * K) % 8 == 0)
                        ncls = max(2, for_c, for_a)
                    else:
                        ncls = 8
                    a_rows = 128
                    if c.srcA == 3 and c.cluster == 1:
                        a_rows = min(128, -(-(-(-M // ncls)) // 8) * 8)
                    elif c.cluster == 1 and M < 128:
                        a_rows = -(-M // 8) * 8
                    smem = c.stages * (a_rows * 64 * 2 + -(-bn_cta // 64) * 64 * 64 * 2)
                    assert smem <= 227 * 1024 and 2 <= c.stages <= 15
                    assert 2 * c.BN <= 512 and c.BN % 16 == 0
                    if halo:
                        assert c.BN in (80, 144, 208) and c.srcA == 3 and N % 16 and M >= 16 and c.P_n == -(-N // (c.BN - 16))
                    assert c.P_k <= ((8 if c.BN != 64 else 1) * -(-(-(-K // 8)) // 64) if c.srcB == 3 else -(-(K + (7 if K % 8 else 0)) // 64))
                    # unaligned operands are never handed to TMA directly (row-major: K for A, N for B)
                    if K % 8:
                        assert c.srcA in (1, 3)      # re-pitched copy, or the per-row-class TMA views
                    if c.srcA == 3:
                        assert (K % 8 or halo) and M >= 8
                        # pair tiles of one row class: 256 rows of a class per SM pair; with halo columns 128 or 192 owned ones
                        assert c.family == ab.FAM_UMMA_1CTA or (M >= (32 if halo else 16) and c.BN in ((144, 208) if halo else (128, 256)))
                        assert c.P_m == ncls * -(-M // (128 * c.cluster * ncls))
                    if N % 8:
                        assert c.srcB in (1, 3)      # re-pitched copy, or the per-k-class TMA views
                    if c.srcB == 3:
                        # k classes: A regrouped class-major, BN - 8 output columns per tile; BN = 64 keeps eight
                        # class accumulators per tile, BN = 128 / 256 makes each class a k split
                        assert N % 8 and K >= 64 and c.BN in (64, 128, 256) and (c.family == ab.FAM_UMMA_1CTA or c.BN == 256)
                        assert c.srcA == 1 and c.P_n == -(-N // (c.BN - 8))
                        if c.BN != 64:
                            assert c.P_k % 8 == 0
                if c.family == ab.FAM_SKINNY:
                    assert min(M, N) <= 16
                if c.family == ab.FAM_CLUSTER:
                    # one launch, no workspace: the k splits are the CTAs of the cluster, none without k values,
                    # the whole grid at most two CTAs per SM, the ring inside the shared-memory limit
                    assert c.cluster in (1, 2, 4, 8, 16) and c.P_k == c.cluster and c.workspace_bytes == 0
                    assert (c.BM, c.BN, c.srcA, c.srcB) == (64, 64, 2, 2)
                    k_cta = -(-(-(-K // c.cluster)) // 16) * 16
                    assert (c.cluster - 1) * k_cta < K
                    assert c.P_m * c.P_n * c.cluster <= 2 * 148 and c.grid == c.P_m * c.P_n * c.cluster
                    assert 1 <= c.stages <= 6 and c.stages <= -(-k_cta // 64)
                    assert (c.stages + 2) * 2 * 64 * 144 + 128 <= 227 * 1024
                # taxonomy label follows the predicate (Section 4.2)
                enough = c.P_m * c.P_n >= 148
                assert (c.taxonomy_class in (0, 1)) == enough


def test_forced_plan_round_trips_its_key():
    M, N, K = 512, 768, 4096
    cands = ab.adapt_plan_candidates(M, N, K, ab.BF16)
    seen = set()
    for c in cands:
        assert c.tiling_key not in seen, "keys must identify configurations"
        seen.add(c.tiling_key)
        h = ab.adapt_matmul_plan_forced(M, N, K, ab.BF16, ab.ROW_MAJOR, ab.ROW_MAJOR, c.tiling_key)
        info = ab.adapt_plan_info(h)
        assert info.tiling_key == c.tiling_key
        assert (info.family, info.BM, info.BN, info.stages, info.P_k) == (c.family, c.BM, c.BN, c.stages, c.P_k)
    with pytest.raises(ab.AdaptError) as e:
        ab.adapt_matmul_plan_forced(M, N, K, ab.BF16, ab.ROW_MAJOR, ab.ROW_MAJOR, 0x1234)
    assert e.value.status == ab.ERR_UNSUPPORTED


def test_cluster_family_is_offered_for_small_grids_only_and_its_key_round_trips():
    small = [c for c in ab.adapt_plan_candidates(50, 311, 3000, ab.F16) if c.family == ab.FAM_CLUSTER]
    assert {c.cluster for c in small} == {1, 2, 4, 8, 16}           # 5 tiles x 16 CTAs still fit
    for c in small:
        info = ab.adapt_plan_info(ab.adapt_matmul_plan_forced(50, 311, 3000, ab.F16, ab.ROW_MAJOR, ab.ROW_MAJOR, c.tiling_key))
        assert (info.family, info.cluster, info.P_k, info.stages) == (ab.FAM_CLUSTER, c.cluster, c.cluster, c.stages)
    assert not [c for c in ab.adapt_plan_candidates(4096, 4096, 64, ab.F16) if c.family == ab.FAM_CLUSTER]
    # a problem of a few tiles and a few hundred k values, unaligned everywhere: the one-launch kernel is the pick
    pick = ab.adapt_plan_info(ab.adapt_matmul_plan(50, 311, 453, ab.F16))
    assert pick.family == ab.FAM_CLUSTER and pick.workspace_bytes == 0


def test_ring_of_a_tile_without_pieces_is_reported_as_launched():
    """Two groups of warps take alternate stages of 64 k values from K = 65 on, with up to three stages each; the key stays loadable."""
    for K in (1, 64, 65, 128, 129, 256, 300, 384, 385, 1000, 5000):
        c = next(c for c in ab.adapt_plan_candidates(70, 90, K, ab.F16) if c.family == ab.FAM_CLUSTER and c.cluster == 1)
        assert c.stages == (1 if K <= 64 else min(3, -(-K // 128))), K
        forced = ab.adapt_plan_info(ab.adapt_matmul_plan_forced(70, 90, K, ab.F16, ab.ROW_MAJOR, ab.ROW_MAJOR, c.tiling_key))
        assert (forced.tiling_key, forced.stages) == (c.tiling_key, c.stages)


def test_split_k_is_chosen_for_small_mn_large_k_and_not_for_large_mn():
    small = ab.adapt_plan_info(ab.adapt_matmul_plan(256, 256, 262144, ab.BF16))
    assert small.P_k > 1 and small.taxonomy_class in (2, 3)
    large = ab.adapt_plan_info(ab.adapt_matmul_plan(8192, 8192, 8192, ab.BF16))
    assert large.P_k == 1 and large.taxonomy_class in (0, 1)
    assert large.family in (ab.FAM_UMMA_1CTA, ab.FAM_UMMA_2CTA)


def test_plan_is_deterministic_across_processes():
    import subprocess
    import sys
    code = ("from paper_2608_10803_b200 import binding as ab;"
            "print([ab.adapt_plan_info(ab.adapt_matmul_plan(*s, 0)).tiling_key for s in "
            "[(7409,156,19633),(1657,12995,164),(64,1024,1024)]])")
    outs = {subprocess.run([sys.executable, "-c", code], cwd=ROOT, capture_output=True, text=True, check=True).stdout
            for _ in range(2)}
    assert len(outs) == 1


def test_cached_plan_lookup_is_fast():
    """Dispatch target: a cached plan costs well under 2 microseconds (measured through ctypes,
    whose own call overhead dominates; the C-level figure is reported by bench.py)."""
    lib = ab.load()
    shapes = synth.sweep_shapes()[:256]
    for (M, N, K) in shapes:
        ab.adapt_matmul_plan(M, N, K, ab.F16)
    f = lib.adapt_matmul_plan
    t0 = time.perf_counter()
    reps = 20
    for _ in range(reps):
        for (M, N, K) in shapes:
            f(M, N, K, 0, 0, 0)
    per_call = (time.perf_counter() - t0) / (reps * len(shapes))
    assert per_call < 5e-6, per_call


def test_sweep_csv_matches_recipe():
    shapes, draws = synth.draw_sweep_shapes()
    assert draws == 2107
    assert shapes == synth.sweep_shapes()
    assert shapes[:5] == [(7409, 156, 19633), (3067, 2, 75528), (6392, 8517, 4), (178, 71, 43035), (1657, 12995, 164)]
    assert len(synth.sweep_oracle_subset()) == 200


# ---- the persisted offline table (Section 3.2: explore offline, look up online) ---------------------

def test_plan_table_round_trip_and_override(tmp_path):
    """Plans saved to a table come back with the same TilingKeys in a fresh cache; a table may name any legal
    configuration of a shape (not only the model's pick) and the online lookup then returns exactly that one;
    lines that are not legal for their shape are skipped; a shape that already has a plan keeps it."""
    ab.adapt_shutdown()
    shapes = [(1000, 1024, 1024, ab.F16), (7, 1024, 1024, ab.F16), (131, 77, 259, ab.BF16), (4096, 4096, 512, ab.BF16),
              (3, 256, 87087, ab.F16), ((1 << 20) + 3, 8, 24, ab.BF16)]
    handles = ab.adapt_plan_many(shapes)
    assert all(handles)
    keys = [ab.adapt_plan_info(h).tiling_key for h in handles]
    ab.adapt_matmul_plan(0, 5, 5, ab.F16)            # no-op and zero-fill plans are not part of the table
    ab.adapt_matmul_plan(5, 5, 0, ab.F16)
    path = str(tmp_path / "plans.txt")
    assert ab.adapt_plan_table_save(path) == len(shapes)

    ab.adapt_shutdown()
    assert ab.adapt_plan_cache_size() == 0
    assert ab.adapt_plan_table_load(path) == len(shapes)
    assert ab.adapt_plan_cache_size() == len(shapes)
    for sh, k in zip(shapes, keys):
        assert ab.adapt_plan_info(ab.adapt_matmul_plan(*sh)).tiling_key == k
    assert ab.adapt_plan_cache_size() == len(shapes)  # every lookup was a hit
    assert ab.adapt_plan_table_load(path) == 0        # shapes that have a plan keep it

    # a hand-written table: the second-best configuration of one shape, one illegal key, one malformed line
    ab.adapt_shutdown()
    M, N, K, dt = 1000, 1024, 1024, ab.F16
    cands = ab.adapt_plan_candidates(M, N, K, dt)
    second = cands[1]
    assert second.tiling_key != cands[0].tiling_key
    lines = open(path).read().splitlines()
    with open(path, "w") as f:
        f.write(lines[0] + "\n")
        f.write(f"{M} {N} {K} {dt} 0 0 {second.tiling_key:016x}\n")
        f.write(f"64 64 64 0 0 0 {second.tiling_key:016x}\n")     # a 1000-row plan's key on a 64^3 shape: stages / P_k do not fit
        f.write("this is not a plan\n")
        f.write(f"-5 64 64 0 0 0 {second.tiling_key:016x}\n")
    n = ab.adapt_plan_table_load(path)
    assert n in (1, 2)
    assert ab.adapt_plan_info(ab.adapt_matmul_plan(M, N, K, dt)).tiling_key == second.tiling_key

    # not a table of this library
    with open(path, "w") as f:
        f.write("# some other file\n1 2 3\n")
    with pytest.raises(ab.AdaptError):
        ab.adapt_plan_table_load(path)
    with pytest.raises(ab.AdaptError):
        ab.adapt_plan_table_load(str(tmp_path / "missing.txt"))
    ab.adapt_shutdown()


def test_calibration_constants_round_trip_and_steer_the_model():
    """The model's machine constants can be read and set by name; a plan made afterwards uses the new value
    (halving the HBM rate makes a memory-bound shape's prediction longer), and unknown names are refused."""
    names = ab.adapt_calibration_names()
    assert "hbm_bw" in names and "launch_us" in names and len(names) == len(set(names)) >= 40
    M, N, K, dt = 40000, 8, 40000, ab.F16         # memory-bound: 3.2 GB of A against 26 GFLOP
    before = min(c.predicted_us for c in ab.adapt_plan_candidates(M, N, K, dt))
    old = ab.adapt_get_calibration("hbm_bw")
    try:
        ab.adapt_set_calibration("hbm_bw", old / 2)
        assert ab.adapt_get_calibration("hbm_bw") == old / 2
        after = min(c.predicted_us for c in ab.adapt_plan_candidates(M, N, K, dt))
        assert after > 1.3 * before
    finally:
        ab.adapt_set_calibration("hbm_bw", old)
    assert min(c.predicted_us for c in ab.adapt_plan_candidates(M, N, K, dt)) == before
    with pytest.raises(ab.AdaptError) as e:
        ab.adapt_set_calibration("no_such_constant", 1.0)
    assert e.value.status == ab.ERR_INVALID_ARG
    with pytest.raises(ab.AdaptError):
        ab.adapt_set_calibration("hbm_bw", float("nan"))


def test_calibrate_fit_improves_or_keeps_the_regret_on_its_own_input(tmp_path):
    """The fitting tool on a small synthetic table of timed configurations: times made from the model's own
    predictions with one constant changed are explained again by moving that constant (the regret it reports
    does not get worse, and the constant moves in the right direction)."""
    import csv as _csv
    from paper_2608_10803_b200 import calibrate
    shapes = [(3000, 3000, 3000, 0), (5000, 40, 20000, 1), (64, 6000, 9000, 0), (9000, 9000, 24, 1), (300, 300, 30000, 0)]
    old = ab.adapt_get_calibration("hbm_bw")
    path = tmp_path / "cand.csv"
    try:
        ab.adapt_set_calibration("hbm_bw", old * 0.8)          # the "machine": a slower memory system
        with open(path, "w", newline="") as f:
            w = _csv.writer(f)
            w.writerow("M,N,K,dtype,family,BN,stages,P_k,cluster,fused,streamk,srcA,srcB,pred_us,t_pro,t_main,t_epi,time_us".split(","))
            for (M, N, K, dt) in shapes:
                for c in ab.adapt_plan_candidates(M, N, K, dt)[:60]:
                    w.writerow([M, N, K, dt, ab.FAMILY_NAMES[c.family], c.BN, c.stages, c.P_k, c.cluster, c.fused, c.streamk, c.srcA, c.srcB,
                                0, 0, 0, 0, f"{c.predicted_us:.4f}"])
        ab.adapt_set_calibration("hbm_bw", old)
        ts = calibrate.TimedSet([str(path)])
        m0 = ts.metrics(ab)
        calibrate.fit([str(path), "--only", "hbm_bw"])
        m1 = ts.metrics(ab)
        assert m1["mean"] <= m0["mean"] + 1e-9 and m1["rms_log_error_near_best"] <= m0["rms_log_error_near_best"] + 1e-9
        assert ab.adapt_get_calibration("hbm_bw") <= old
    finally:
        ab.adapt_set_calibration("hbm_bw", old)
