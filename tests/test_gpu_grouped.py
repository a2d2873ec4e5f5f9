"""Grouped launches: lists of small GEMMs and strided batches that leave as one launch give the bits of the calls made alone
(lists), and the oracle's exact result on integers (strided batches)."""
import random

import numpy as np
import pytest
import torch

from oracle import gemm as og
from paper_2608_10803_b200 import binding as ab
from paper_2608_10803_b200 import synth

from gpu_util import init

pytestmark = pytest.mark.gpu


def stream():
    return torch.cuda.current_stream().cuda_stream


def offset_operand(rows, cols, seed, dtype, offset):
    """A dense operand whose first element sits `offset` elements behind an aligned address."""
    flat = torch.empty(rows * cols + offset, dtype=synth.torch_dtype(dtype), device="cuda")
    flat[offset:] = synth.draw_operand(rows, cols, synth.U11, seed, dtype, "cuda").reshape(-1)
    return flat[offset:]


@pytest.mark.parametrize("layouts", [(0, 0), (0, 1), (1, 0), (1, 1)])
@pytest.mark.parametrize("offset", [0, 1, 8])
def test_grouped_list_gives_the_bits_of_single_calls(layouts, offset):
    """Every split of the one-launch plans (1 to 16 pieces), CUDA-core plans, tile edges, both types in one list, and a list
    longer than one launch takes."""
    init()
    r = random.Random(5 + offset)
    dims = [1, 3, 16, 33, 63, 64, 65, 100, 128, 200, 257]
    shapes = [(r.choice(dims), r.choice(dims), r.choice([1, 5, 16, 31, 64, 65, 130, 250, 400, 787, 1014])) for _ in range(90)]
    shapes += [(64, 64, 1024), (17, 30, 900), (65, 129, 513), (4, 1000, 1000), (300, 300, 64)]
    calls = []
    for i, (M, N, K) in enumerate(shapes):
        dt = ab.F16 if i % 3 else ab.BF16
        A, B = offset_operand(M, K, 2 * i, dt, offset), offset_operand(K, N, 2 * i + 1, dt, offset)
        C1, C2 = (torch.full((M * N + offset,), float("nan"), dtype=A.dtype, device="cuda")[offset:] for _ in range(2))
        calls.append((ab.adapt_matmul_plan(M, N, K, dt, *layouts), A, B, C1, C2))
    for p, A, B, C1, _ in calls:
        ab.adapt_matmul(p, A.data_ptr(), B.data_ptr(), C1.data_ptr(), stream())
    torch.cuda.synchronize()
    launches = ab.adapt_launch_count()
    ab.adapt_matmul_batch([c[0] for c in calls], *([c[j].data_ptr() for c in calls] for j in (1, 2, 4)), stream())
    torch.cuda.synchronize()
    assert ab.adapt_launch_count() - launches < len(calls) // 2
    ab.adapt_poll_device_status(stream())
    pieces = set()
    for (p, _, _, C1, C2), shape in zip(calls, shapes):
        pieces.add(ab.adapt_plan_info(p).cluster)
        assert torch.equal(C1.view(torch.int16), C2.view(torch.int16)), shape
    assert {1, 4, 8} <= pieces


@pytest.mark.parametrize("layouts", [(0, 0), (0, 1), (1, 0), (1, 1)])
@pytest.mark.parametrize("dtype", [ab.F16, ab.BF16])
def test_tiles_shared_by_several_ctas_give_the_bits_of_single_calls(layouts, dtype):
    """Short lists whose longest k chains are shared by two CTAs (four pieces) or four (eight, sixteen), beside tiles that are not; ragged
    last pieces, odd numbers of shared tiles, tiles of one row and column, and a list that only holds shared tiles."""
    init()
    lists = [[(84, 39, 1014), (20, 30, 40)], [(504, 209, 576), (100, 100, 100), (30, 7, 20)], [(64, 64, 1024), (65, 63, 1000), (17, 763, 618), (105, 845, 611), (1, 1, 500)],
             [(38, 48, 787), (48, 38, 808), (1, 70, 790)], [(64, 128, 1008), (16, 200, 520), (129, 1, 400), (300, 200, 50), (10, 10, 65), (33, 65, 130), (7, 9, 11), (40, 342, 267)]]
    seen = set()
    for k, shapes in enumerate(lists):
        calls = []
        for i, (M, N, K) in enumerate(shapes):
            p = ab.adapt_matmul_plan(M, N, K, dtype, *layouts)
            assert ab.adapt_plan_info(p).family in (ab.FAM_CLUSTER, ab.FAM_SIMT), (M, N, K)
            seen.add(ab.adapt_plan_info(p).cluster)
            A, B = offset_operand(M, K, 900 + 2 * i, dtype, i % 3), offset_operand(K, N, 901 + 2 * i, dtype, k % 2)
            calls.append((p, A, B) + tuple(torch.full((M * N,), float("nan"), dtype=A.dtype, device="cuda") for _ in range(2)))
        for p, A, B, C1, _ in calls:
            ab.adapt_matmul(p, A.data_ptr(), B.data_ptr(), C1.data_ptr(), stream())
        launches = ab.adapt_launch_count()
        ab.adapt_matmul_batch([c[0] for c in calls], *([c[j].data_ptr() for c in calls] for j in (1, 2, 4)), stream())
        assert ab.adapt_launch_count() - launches == 1
        torch.cuda.synchronize()
        ab.adapt_poll_device_status(stream())
        for (_, _, _, C1, C2), shape in zip(calls, shapes):
            assert torch.equal(C1.view(torch.int16), C2.view(torch.int16)), shape
    assert {1, 4, 8, 16} <= seen


def test_grouped_list_keeps_the_order_of_dependent_calls():
    """Calls that read what an earlier call of the list wrote, overwrite what it read, or write the same output."""
    init()
    n, dt = 96, ab.F16
    plan = ab.adapt_matmul_plan(n, n, n, dt)
    eye = torch.eye(n, dtype=torch.float16, device="cuda")
    X = [synth.position_coded(n, n, dt, 3, "cuda").contiguous() for _ in range(2)] + [torch.zeros((n, n), dtype=torch.float16, device="cuda") for _ in range(3)]
    roll = torch.roll(eye, 1, 1).contiguous()
    # X2 = X0 R, X3 = X2 R, X0 = X1 I (overwrites an input), X4 = X0 R, X4 = X3 I (overwrites an output)
    steps = [(0, roll, 2), (2, roll, 3), (1, eye, 0), (0, roll, 4), (3, eye, 4)]
    want = [x.clone() for x in X]
    for a, b, c in steps:
        want[c] = want[a] @ b
    ab.adapt_matmul_batch([plan] * 5, [X[a].data_ptr() for a, _, _ in steps], [b.data_ptr() for _, b, _ in steps],
                          [X[c].data_ptr() for _, _, c in steps], stream())
    torch.cuda.synchronize()
    for x, w in zip(X, want):
        assert torch.equal(x, w)


def test_grouped_list_enqueues_the_calls_before_a_refused_one():
    init()
    plan = ab.adapt_matmul_plan(40, 24, 32, ab.F16)
    A, B = torch.ones((40, 32), dtype=torch.float16, device="cuda"), torch.ones((32, 24), dtype=torch.float16, device="cuda")
    C = torch.zeros((3, 40, 24), dtype=torch.float16, device="cuda")
    with pytest.raises(ab.AdaptError) as e:
        ab.adapt_matmul_batch([plan] * 3, [A.data_ptr()] * 3, [B.data_ptr(), 0, B.data_ptr()], [C[i].data_ptr() for i in range(3)], stream())
    torch.cuda.synchronize()
    assert e.value.status == ab.ERR_INVALID_ARG and bool((C[0] == 32).all()) and not C[1:].any()


def check_strided(M, N, K, batch, dtype, lA=0, lB=0, shared_a=False, shared_b=False, gap=(0, 0, 0), offset=0, plan=None):
    init()
    na, nb, nc = M * K + gap[0], K * N + gap[1], M * N + gap[2]
    def operand(count, each, seed):
        flat = torch.empty(count * each + offset, dtype=synth.torch_dtype(dtype), device="cuda")
        flat[offset:] = synth.draw_operand(count, each, ("integer", -4, 4), seed, dtype, "cuda").reshape(-1)
        return flat[offset:]
    A, B = operand(1 if shared_a else batch, na, 71), operand(1 if shared_b else batch, nb, 72)
    C = torch.full((batch * nc + offset,), 77.0, dtype=A.dtype, device="cuda")[offset:]
    plan = plan or ab.adapt_matmul_plan(M, N, K, dtype, lA, lB)
    ab.adapt_matmul_strided_batch(plan, A.data_ptr(), 0 if shared_a else na, B.data_ptr(), 0 if shared_b else nb, C.data_ptr(), nc, batch, stream())
    torch.cuda.synchronize()
    ab.adapt_poll_device_status(stream())
    for b in range(batch):
        a_, b_ = A[0 if shared_a else b * na:][:M * K], B[0 if shared_b else b * nb:][:K * N]
        _, C16 = og.gemm(synth.bits(a_), synth.bits(b_), M, N, K, dtype, lA, lB)
        got = C[b * nc:(b + 1) * nc]
        assert np.array_equal(synth.bits(got[:M * N]).reshape(C16.shape), C16), (M, N, K, b)
        assert bool((got[M * N:] == 77).all()), "the gap between two outputs was written"


@pytest.mark.parametrize("dtype", [ab.F16, ab.BF16])
@pytest.mark.parametrize("shape", [(128, 128, 64, 5), (64, 64, 64, 3), (65, 33, 130, 7), (8, 8, 8, 40), (1, 1, 1, 9), (16, 264, 96, 6), (129, 257, 72, 4),
                                   (40, 1000, 200, 3), (256, 128, 520, 2), (48, 80, 1024, 2), (320, 192, 128, 9), (8, 17, 33, 300)])
def test_strided_batch_exact_in_every_layout(shape, dtype):
    M, N, K, batch = shape
    for lA, lB in ((0, 0), (0, 1), (1, 0), (1, 1)):
        check_strided(M, N, K, batch, dtype, lA, lB)
    check_strided(M, N, K, batch, dtype, shared_b=True, gap=(3, 0, 5))
    check_strided(M, N, K, batch, dtype, 0, 1, shared_a=True, gap=(0, 8, 16))
    check_strided(M, N, K, batch, dtype, gap=(1, 1, 1), offset=1)


def test_strided_batch_whose_entries_feed_one_another_runs_in_order():
    """Entry i writes the operand that entry i + 1 reads."""
    init()
    n, batch = 64, 6
    X = torch.zeros((batch + 1, n, n), dtype=torch.float16, device="cuda")
    X[0] = synth.position_coded(n, n, ab.F16, 3, "cuda")
    roll = torch.roll(torch.eye(n, dtype=torch.float16, device="cuda"), 1, 1).contiguous()
    plan = ab.adapt_matmul_plan(n, n, n, ab.F16)
    ab.adapt_matmul_strided_batch(plan, X.data_ptr(), n * n, roll.data_ptr(), 0, X[1].data_ptr(), n * n, batch, stream())
    torch.cuda.synchronize()
    for i in range(batch):
        assert torch.equal(X[i + 1], X[i] @ roll)


def installed_plans(tmp_path, shapes, want):
    """Plans of a table that names, for every (M, N, K, dtype), the first candidate that `want` accepts."""
    path = tmp_path / "plans.txt"
    assert ab.adapt_plan_table_save(str(path)) >= 0
    lines = [path.read_text().splitlines()[0]]
    for M, N, K, dt in shapes:
        c = next(c for c in ab.adapt_plan_candidates(M, N, K, dt) if want(c))
        lines.append(f"{M} {N} {K} {dt} 0 0 {c.tiling_key:016x}")
    path.write_text("\n".join(lines) + "\n")
    assert ab.adapt_plan_table_load(str(path)) == len(shapes), "a shape had a plan before"
    return [ab.adapt_matmul_plan(*s) for s in shapes]


@pytest.mark.parametrize("pieces", [2, 4])
def test_list_of_short_k_plans_that_a_table_cut_into_pieces(tmp_path, pieces):
    """All K <= 64, so that nothing but the number of pieces tells the launch which kernel it needs."""
    ab.adapt_shutdown()
    init()
    shapes = [(128, 128, 64, ab.F16), (65, 127, 64, ab.F16), (61, 200, 63, ab.F16)] + ([(128, 64, 32, ab.F16), (3, 70, 48, ab.F16)] if pieces == 2 else [])
    plans = installed_plans(tmp_path, shapes, lambda c: c.family == ab.FAM_CLUSTER and c.cluster == pieces)
    A = [synth.draw_operand(M, K, synth.U11, 2 * i, dt, "cuda") for i, (M, N, K, dt) in enumerate(shapes)]
    B = [synth.draw_operand(K, N, synth.U11, 2 * i + 1, dt, "cuda") for i, (M, N, K, dt) in enumerate(shapes)]
    alone, listed = ([torch.full((M, N), float("nan"), dtype=torch.float16, device="cuda") for M, N, _, _ in shapes] for _ in range(2))
    for p, a, b, c in zip(plans, A, B, alone):
        ab.adapt_matmul(p, a.data_ptr(), b.data_ptr(), c.data_ptr(), stream())
    before = ab.adapt_launch_count()
    ab.adapt_matmul_batch(plans, *([t.data_ptr() for t in x] for x in (A, B, listed)), stream())
    torch.cuda.synchronize()
    ab.adapt_poll_device_status(stream())
    assert ab.adapt_launch_count() - before == 1
    for x, y, s in zip(alone, listed, shapes):
        assert torch.equal(x.view(torch.int16), y.view(torch.int16)), s
    ab.adapt_shutdown()


def strided_and_alone(plan, M, N, K, dtype, batch, offset=0, seed=31):
    """The same batch in one call and entry by entry, with non-integer operands; launches of the one call."""
    A = offset_operand(batch * M, K, seed, dtype, offset)
    B = offset_operand(batch * K, N, seed + 1, dtype, offset)
    one, many = (torch.full((batch * M * N,), float("nan"), dtype=A.dtype, device="cuda") for _ in range(2))
    for e in range(batch):
        ab.adapt_matmul(plan, A.data_ptr() + 2 * e * M * K, B.data_ptr() + 2 * e * K * N, many.data_ptr() + 2 * e * M * N, stream())
    before = ab.adapt_launch_count()
    ab.adapt_matmul_strided_batch(plan, A.data_ptr(), M * K, B.data_ptr(), K * N, one.data_ptr(), M * N, batch, stream())
    launches = ab.adapt_launch_count() - before
    torch.cuda.synchronize()
    ab.adapt_poll_device_status(stream())
    return A, B, one, many, launches


@pytest.mark.parametrize("offset", [0, 1])
@pytest.mark.parametrize("table", [False, True])
def test_strided_batch_keeps_a_configuration_that_was_asked_for(tmp_path, table, offset):
    """Every kind of candidate, forced or named by a plan table: the bits of the entries alone."""
    M, N, K, batch, dt = 96, 200, 1000, 12, ab.F16
    init()
    kinds = {}
    for c in ab.adapt_plan_candidates(M, N, K, dt):
        kinds.setdefault((c.family, c.cluster, c.P_k > 1, c.fused, c.srcA, c.srcB), c)
    assert {c.cluster for c in kinds.values() if c.family == ab.FAM_CLUSTER} == {1, 2, 4, 8, 16}
    for c in kinds.values():
        if table:
            ab.adapt_shutdown()
            init()
            plan, = installed_plans(tmp_path, [(M, N, K, dt)], lambda x: x.tiling_key == c.tiling_key)
        else:
            plan = ab.adapt_matmul_plan_forced(M, N, K, dt, 0, 0, c.tiling_key)
        assert ab.adapt_plan_info(plan).tiling_key == c.tiling_key
        if table and c.tiling_key == ab.adapt_plan_candidates(M, N, K, dt)[0].tiling_key:
            continue                                                    # what the library would choose itself
        _, _, one, many, launches = strided_and_alone(plan, M, N, K, dt, batch, offset)
        assert torch.equal(one.view(torch.int16), many.view(torch.int16)), (ab.FAMILY_NAMES[c.family], c.cluster, c.P_k, c.BN)
        assert launches == 1 or c.family != ab.FAM_CLUSTER
    if table:
        ab.adapt_shutdown()


@pytest.mark.parametrize("shape", [(96, 200, 1000, 12, 1), (130, 77, 259, 200, 2), (128, 256, 512, 160, 1), (513, 96, 64, 100, 1)])
@pytest.mark.parametrize("dtype", [ab.F16, ab.BF16])
def test_strided_batch_of_a_chosen_plan_rounds_once_and_repeats(shape, dtype):
    """One or two launches, every element within one rounding of the 16-bit result (and an fp32 sum's error), the same bits again."""
    M, N, K, batch, most = shape
    init()
    plan = ab.adapt_matmul_plan(M, N, K, dtype)
    A, B, one, many, launches = strided_and_alone(plan, M, N, K, dtype, batch)
    assert launches <= most
    again = strided_and_alone(plan, M, N, K, dtype, batch)[2]
    assert torch.equal(one.view(torch.int16), again.view(torch.int16))
    a, b = A.view(batch, M, K).double(), B.view(batch, K, N).double()
    want, scale = torch.bmm(a, b), torch.bmm(a.abs(), b.abs())
    # fp32 products are exact; a sum of K of them in any order, truncated at each step, is within K 2^-23 of the sum of magnitudes; then one
    # rounding to 16 bits
    half_ulp = 2.0 ** -11 if dtype == ab.F16 else 2.0 ** -8
    bound = half_ulp * want.abs() + (K * 2.0 ** -23) * 1.01 * scale + 2.0 ** -25
    for got in (one, many):
        assert bool(((got.view(batch, M, N).double() - want).abs() <= bound).all())


def test_alternating_types_and_layouts_fill_their_launches():
    """Calls of four variants in turn: one launch per 64 calls of a variant."""
    init()
    M, N, K = 24, 40, 56
    variants = [(ab.F16, 0, 0), (ab.BF16, 0, 0), (ab.F16, 0, 1), (ab.BF16, 1, 0)]
    plans = [ab.adapt_matmul_plan(M, N, K, *v) for v in variants]
    X = [[synth.draw_operand(r, c, ("integer", -4, 4), 40 + j, v[0], "cuda") for j, (r, c) in enumerate(((M, K), (K, N)))] for v in variants]
    C = torch.zeros((512, M, N), dtype=torch.float16, device="cuda")
    before = ab.adapt_launch_count()
    ab.adapt_matmul_batch([plans[i % 4] for i in range(512)], *([X[i % 4][j].data_ptr() for i in range(512)] for j in (0, 1)),
                          [C[i].data_ptr() for i in range(512)], stream())
    torch.cuda.synchronize()
    assert ab.adapt_launch_count() - before == 8
    for i in (0, 1, 2, 3, 255, 510, 511):
        dt, lA, lB = variants[i % 4]
        _, want = og.gemm(synth.bits(X[i % 4][0]).reshape(-1), synth.bits(X[i % 4][1]).reshape(-1), M, N, K, dt, lA, lB)
        assert np.array_equal(C[i].view(torch.int16).cpu().numpy().view(np.uint16).reshape(want.shape), want), i


@pytest.mark.parametrize("dtype", [ab.F16, ab.BF16])
@pytest.mark.parametrize("shape", [(65, 33, 70), (17, 130, 63), (100, 64, 8), (64, 200, 400), (130, 264, 328)])
def test_special_values_stay_in_their_rows_columns_and_entries(shape, dtype):
    """Infinities and NaN at the ends of rows and k ranges, in lists and strided batches, aligned and not: only the outputs that they
    belong to are touched, and those as the arithmetic gives them."""
    M, N, K = shape
    init()
    batch = 24
    A, B = (synth.draw_operand(batch * r, c, ("integer", 1, 3), seed, dtype, "cuda").view(batch, r, c) for r, c, seed in ((M, K, 81), (K, N, 82)))
    for e in range(0, batch, 3):
        A[e, M - 1, K - 1], A[e, 0, 0], B[e, K - 1, N - 1], A[e, 5, K // 2] = float("inf"), float("-inf"), float("inf"), float("nan")
    want = torch.bmm(A.double(), B.double()).to(A.dtype)                # small integers: exact before the one rounding
    plan = ab.adapt_matmul_plan(M, N, K, dtype)
    for offset in (0, 1):
        a, b = (torch.empty(x.numel() + offset, dtype=A.dtype, device="cuda")[offset:].copy_(x.reshape(-1)) for x in (A, B))
        listed, strided = (torch.full((batch, M, N), 7.0, dtype=A.dtype, device="cuda") for _ in range(2))
        ab.adapt_matmul_batch([plan] * batch, [a.data_ptr() + 2 * e * M * K for e in range(batch)], [b.data_ptr() + 2 * e * K * N for e in range(batch)],
                              [listed[e].data_ptr() for e in range(batch)], stream())
        ab.adapt_matmul_strided_batch(plan, a.data_ptr(), M * K, b.data_ptr(), K * N, strided.data_ptr(), M * N, batch, stream())
        torch.cuda.synchronize()
        ab.adapt_poll_device_status(stream())
        for got in (listed, strided):
            assert torch.equal(torch.isnan(got), torch.isnan(want)) and torch.equal(torch.where(torch.isnan(got), 0.0, got.float()), torch.where(torch.isnan(want), 0.0, want.float()))
