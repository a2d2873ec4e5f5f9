"""Tall pair tiles (512 x 256 outputs per SM pair): bit-exact on integers at the edges of tiles, k ranges and schedules, in every layout, with
row classes, with the fused add, and on buffers that send the plan to other tiles."""
import numpy as np
import pytest
import torch

from oracle import gemm as og
from paper_2608_10803_b200 import binding as ab
from paper_2608_10803_b200 import synth

from gpu_util import init, sample_rows

pytestmark = pytest.mark.gpu


def tall_plan(M, N, K, dtype, lA=0, lB=0):
    for c in ab.adapt_plan_candidates(M, N, K, dtype, lA, lB):
        if c.BM == 512:
            return ab.adapt_matmul_plan_forced(M, N, K, dtype, lA, lB, c.tiling_key)
    raise AssertionError(f"no tall candidate for {M}x{N}x{K}")


def integers(rows, cols, seed, dtype, offset=0):
    flat = synth.draw_operand(1, rows * cols + offset, ("integer", -3, 3), seed, dtype, "cuda").reshape(-1)
    return flat[offset:]


def check(M, N, K, dtype, lA=0, lB=0, addmm=None, offsets=(0, 0, 0), rows=None, d_offset=0):
    init()
    plan = tall_plan(M, N, K, dtype, lA, lB)
    oa, ob, oc = offsets
    A, B = integers(M, K, 1, dtype, oa), integers(K, N, 2, dtype, ob)
    C = torch.full((M * N + oc + 64,), float("nan"), dtype=synth.torch_dtype(dtype), device="cuda")
    guard = synth.bits(C).copy()
    st = torch.cuda.current_stream().cuda_stream
    D = None
    if addmm:
        D = integers(1 if addmm == "bias" else M, N, 3, dtype, d_offset)
        ab.adapt_addmm(plan, A.data_ptr(), B.data_ptr(), D.data_ptr(), addmm == "bias", 2.0, -1.0, C.data_ptr() + 2 * oc, st)
    else:
        ab.adapt_matmul(plan, A.data_ptr(), B.data_ptr(), C.data_ptr() + 2 * oc, st)
    torch.cuda.synchronize()
    ab.adapt_poll_device_status(st)
    got = synth.bits(C)
    rows = np.arange(M) if rows is None else rows
    a = (A.reshape(K, M).t() if lA else A.reshape(M, K)).double().cpu().numpy()[rows]
    b = (B.reshape(N, K).t() if lB else B.reshape(K, N)).double().cpu().numpy()
    want = a @ b                                        # integers below 2^53: exact in any order
    if D is not None:
        d = D.double().cpu().numpy()
        want = 2.0 * want - (d[None, :] if addmm == "bias" else d.reshape(M, N)[rows])
    want = synth.bits(torch.from_numpy(want).to(synth.torch_dtype(dtype))).reshape(len(rows), N)   # |sum| < 2^24: one rounding
    body = got.reshape(-1)[oc:oc + M * N].reshape(M, N)[rows]
    assert np.array_equal(body, want), (M, N, K, lA, lB, addmm, int((body != want).sum()))
    flat = got.reshape(-1)
    assert np.array_equal(flat[:oc], guard.reshape(-1)[:oc]) and np.array_equal(flat[oc + M * N:], guard.reshape(-1)[oc + M * N:]), "written outside C"


# one k-block beyond the first, around the distance between the halves and the ring, and long; ragged ends of every dimension
@pytest.mark.parametrize("K", [72, 128, 136, 192, 200, 256, 264, 328, 448, 520, 1000])
@pytest.mark.parametrize("dtype", [ab.F16, ab.BF16])
def test_k_ranges(K, dtype):
    check(512, 256, K, dtype)
    check(1000, 272, K, dtype)


@pytest.mark.parametrize("lA", [0, 1])
@pytest.mark.parametrize("lB", [0, 1])
@pytest.mark.parametrize("addmm", [None, "bias", "matrix"])
def test_layouts_edges_and_fused_add(lA, lB, addmm):
    # (a matrix D: tall tiles from K = 1024 on)
    for M, N, K in [(257, 16, 80), (264, 144, 328), (512, 512, 264), (776, 240, 392), (1288, 1040, 136), (300, 272, 1032), (1288, 528, 1096)]:
        check(M, N, K, ab.BF16 if lA else ab.F16, lA, lB, addmm)


# row classes: K off 16-byte boundaries; an odd number of 2048-row groups, a last group of a few rows
@pytest.mark.parametrize("shape", [(2056, 256, 203), (4096, 272, 131), (4500, 688, 333), (6150, 64, 517), (9000, 48, 75), (4500, 80, 1037)])
@pytest.mark.parametrize("addmm", [None, "matrix"])
def test_row_classes(shape, addmm):
    M, N, K = shape
    check(M, N, K, ab.F16, addmm=addmm)


# several waves of tiles; leftovers cut into halves; an odd row of blocks beside whole waves
@pytest.mark.parametrize("shape", [(4096, 4864, 72), (20000, 1024, 136), (19200, 1280, 72), (38400, 264 - 8, 72), (30000, 1360, 200)])
def test_schedules(shape):
    M, N, K = shape
    check(M, N, K, ab.F16, rows=sample_rows(M, 600))


def test_rows_before_a_class_view_do_not_leak():
    """An infinity at the end of a row sits in front of the next row's view."""
    M, N, K, dt = 4100, 128, 139, ab.F16
    init()
    plan = tall_plan(M, N, K, dt)
    A, B = integers(M, K, 5, dt).reshape(M, K).clone(), integers(K, N, 6, dt)
    A[::3, K - 1] = float("inf")
    C = torch.empty(M, N, dtype=torch.float16, device="cuda")
    st = torch.cuda.current_stream().cuda_stream
    ab.adapt_matmul(plan, A.data_ptr(), B.data_ptr(), C.data_ptr(), st)
    torch.cuda.synchronize()
    finite = torch.isfinite(C).all(dim=1).cpu().numpy()
    assert finite[1::3].all() and finite[2::3].all()
    keep = torch.ones(M, dtype=torch.bool)
    keep[::3] = False
    want = A.cpu()[keep].double() @ B.cpu().reshape(K, N).double()
    assert torch.equal(C.cpu()[keep], want.to(torch.float16))


@pytest.mark.parametrize("offsets", [(0, 0, 8), (0, 0, 1), (8, 0, 0), (1, 8, 0), (3, 5, 16)])
def test_unaligned_buffers(offsets):
    check(700, 272, 200, ab.F16, offsets=offsets)
    check(2500, 272, 203, ab.F16, offsets=offsets)
    for addmm in ("bias", "matrix"):
        check(700, 272, 200, ab.F16, addmm=addmm, offsets=offsets, d_offset=8)
        check(700, 272, 200, ab.F16, addmm=addmm, d_offset=offsets[0] + offsets[1])
