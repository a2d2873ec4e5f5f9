"""Tall pair tiles that are computed whole (512 x 256 outputs, not cut into their 256-row halves): bit-exact on integers for every length of k range
around the lag of the halves and the ring, in every layout and type, with row classes, with a second tile and with single blocks behind them, and
with the fused add, in place and with special values."""
import numpy as np
import pytest
import torch

from oracle import gemm as og
from paper_2608_10803_b200 import binding as ab
from paper_2608_10803_b200 import synth

from gpu_util import init

pytestmark = pytest.mark.gpu

# (M, N) with ragged last tiles.  Plain: 10 x 4 tiles of 512 rows, 10 x 4 and 4 single blocks, 16 x 7 (a second one on some of 74 pairs), 3 x 19 and 19
# single blocks (two of them on some of the other 17 pairs).
# Row classes: 8 x 5, 16 x 7, and 8 x 7 with 56 single blocks.
PLAIN = {"one": (5000, 1008), "odd": (5300, 1008), "two": (8100, 1776), "few": (1771, 4720)}
CLASSES = {"one": (4000, 1264), "two": (8100, 1776), "odd": (6100, 1776)}


def tall_plan(M, N, K, dtype, lA=0, lB=0, classes=False):
    for c in ab.adapt_plan_candidates(M, N, K, dtype, lA, lB):
        if c.BM == 512 and (c.srcA == 3) == classes:
            n = 8 if classes else 1
            blocks, columns = -(-M // (256 * n)), -(-N // 256)
            slots, tiles, single = torch.cuda.get_device_properties(0).multi_processor_count // 2, blocks // 2 * n * columns, blocks % 2 * n * columns
            assert tiles >= slots or 2 * (tiles % slots) + single > slots, "cut into halves: no whole tile"
            assert c.grid == 2 * min(tiles + single, slots)             # (halves of cut tiles would be counted twice)
            return ab.adapt_matmul_plan_forced(M, N, K, dtype, lA, lB, c.tiling_key)
    raise AssertionError(f"no tall candidate for {M}x{N}x{K}")


def integers(n, seed, dtype):
    return synth.draw_operand(1, n, ("integer", -3, 3), seed, dtype, "cuda").reshape(-1)


def check(M, N, K, dtype, lA=0, lB=0, classes=False, addmm=None, in_place=False):
    init()
    plan = tall_plan(M, N, K, dtype, lA, lB, classes)
    A, B = integers(M * K, 1, dtype), integers(K * N, 2, dtype)
    flat = torch.full((M * N + 128,), float("nan"), dtype=A.dtype, device="cuda")
    C = flat[64:64 + M * N]
    st = torch.cuda.current_stream().cuda_stream
    want = (A.view(K, M).t() if lA else A.view(M, K)).double() @ (B.view(N, K).t() if lB else B.view(K, N)).double()
    if addmm:
        D = integers(N if addmm == "bias" else M * N, 3, dtype)
        want = 2.0 * want - (D.double() if addmm == "bias" else D.double().view(M, N))
        if in_place:
            C.copy_(D)
            D = C
        assert ab.adapt_plan_info_call(plan, C.data_ptr(), D.data_ptr(), addmm == "bias").BM == 512
        ab.adapt_addmm(plan, A.data_ptr(), B.data_ptr(), D.data_ptr(), addmm == "bias", 2.0, -1.0, C.data_ptr(), st)
    else:
        assert ab.adapt_plan_info_call(plan, C.data_ptr()).BM == 512
        ab.adapt_matmul(plan, A.data_ptr(), B.data_ptr(), C.data_ptr(), st)
    torch.cuda.synchronize()
    ab.adapt_poll_device_status(st)
    want = want.to(A.dtype)                                             # integers: exact in any order, |sum| < 2^24, one rounding
    wrong = int((C.view(M, N) != want).sum())
    assert wrong == 0, (M, N, K, lA, lB, addmm, in_place, wrong)
    assert torch.isnan(flat[:64]).all() and torch.isnan(flat[64 + M * N:]).all(), "written outside C"


# 2 to 9 and 17 k-blocks of 64, the last one ragged
@pytest.mark.parametrize("blocks", [2, 3, 4, 5, 6, 7, 8, 9, 17])
@pytest.mark.parametrize("dtype", [ab.F16, ab.BF16])
def test_k_blocks(blocks, dtype):
    check(*PLAIN["one"], 64 * blocks - 56, dtype)
    check(*PLAIN["two"], 64 * blocks, dtype)
    check(*CLASSES["one"], 64 * blocks - 59, dtype, classes=True)
    check(*CLASSES["two"], 64 * blocks - 9, dtype, classes=True)


@pytest.mark.parametrize("lA", [0, 1])
@pytest.mark.parametrize("lB", [0, 1])
@pytest.mark.parametrize("addmm", [None, "bias", "matrix"])
def test_layouts_and_fused_add(lA, lB, addmm):
    for where, K in [("one", 1032), ("odd", 1096), ("two", 1032), ("few", 1096)] + ([] if addmm == "matrix" else [("one", 456), ("odd", 72), ("two", 200), ("few", 328)]):
        check(*PLAIN[where], K, ab.BF16 if lA else ab.F16, lA, lB, addmm=addmm)


@pytest.mark.parametrize("where", list(CLASSES))
@pytest.mark.parametrize("addmm", [None, "bias", "matrix"])
def test_row_classes(where, addmm):
    for K, dtype in [(1027, ab.F16), (1093, ab.BF16)] + ([] if addmm == "matrix" else [(331, ab.F16), (142, ab.BF16)]):
        check(*CLASSES[where], K, dtype, classes=True, addmm=addmm)


@pytest.mark.parametrize("classes", [False, True])
@pytest.mark.parametrize("where", ["one", "odd", "two"])
def test_added_matrix_in_place(where, classes):
    check(*(CLASSES if classes else PLAIN)[where], 1027 if classes else 1032, ab.BF16, classes=classes, addmm="matrix", in_place=True)


@pytest.mark.parametrize("classes", [False, True])
@pytest.mark.parametrize("dtype", [ab.F16, ab.BF16])
def test_infinities_nan_and_the_types_largest_values(classes, dtype):
    """Special values of A, B and D reach exactly the outputs that the arithmetic gives."""
    M, N = (CLASSES if classes else PLAIN)["one"]
    K = 1027 if classes else 1032
    init()
    plan = tall_plan(M, N, K, dtype, classes=classes)
    st = torch.cuda.current_stream().cuda_stream
    A, B, D = (synth.draw_operand(r, c, ("integer", 1, 4), seed, dtype, "cuda") for r, c, seed in ((M, K, 61), (K, N, 62), (M, N, 63)))
    inf, nan, big = float("inf"), float("nan"), torch.finfo(A.dtype).max
    D[0, 0], D[M - 1, N - 1], D[M // 2, N // 2], D[1, N - 2], D[2, 3], D[300, 17] = inf, -inf, nan, -big, big, inf
    A[3, K - 1], B[K - 1, N - 3], A[4, 0], A[300, 64], A[M - 1, K - 1] = inf, -inf, nan, -inf, inf
    rows = np.array(sorted({0, 1, 2, 3, 4, 5, 11, 12, 256, 299, 300, 301, 308, M // 2, M - 9, M - 2, M - 1}))
    at = torch.from_numpy(rows).cuda()
    exponent = 0x7C00 if dtype == ab.F16 else 0x7F80
    is_nan = lambda x: ((x & exponent) == exponent) & ((x & (0x7FFF - exponent)) != 0)
    for d in (D, D[M // 2].contiguous()):
        for alpha, beta in ((1.0, 1.0), (-2.0, 0.5), (1.0, 0.0)):
            with np.errstate(all="ignore"):
                _, want = og.addmm_rows(synth.bits(A), synth.bits(B), synth.bits(d), M, N, K, dtype, alpha, beta, rows=rows)
            C = torch.full((M, N), 7.0, dtype=A.dtype, device="cuda")
            ab.adapt_addmm(plan, A.data_ptr(), B.data_ptr(), d.data_ptr(), d.dim() == 1, alpha, beta, C.data_ptr(), st)
            torch.cuda.synchronize()
            ab.adapt_poll_device_status(st)
            got, want = synth.bits(C.index_select(0, at)).reshape(-1).astype(np.uint16), want.reshape(-1).astype(np.uint16)
            assert (is_nan(got) == is_nan(want)).all() and (got == want)[~is_nan(want)].all(), (dtype, classes, alpha, beta, d.dim())
