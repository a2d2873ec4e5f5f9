"""Strided batches on the tensor-core kernel: one launch (and at most one copy) for all entries, bit-exact on integers."""
import numpy as np
import pytest
import torch

from oracle import gemm as og
from paper_2608_10803_b200 import binding as ab
from paper_2608_10803_b200 import synth

from gpu_util import init
from test_gpu_grouped import check_strided

pytestmark = pytest.mark.gpu


@pytest.mark.parametrize("dtype", [ab.F16, ab.BF16])
@pytest.mark.parametrize("shape", [(128, 256, 512, 160), (200, 264, 328, 120), (130, 77, 259, 200), (8, 512, 512, 256), (64, 1000, 520, 100), (513, 96, 64, 100),
                                   (1024, 512, 136, 30), (300, 40, 1000, 100)])
def test_strided_batch_on_the_tensor_core_kernel(shape, dtype):
    M, N, K, batch = shape
    init()
    cases = [dict(lA=lA, lB=lB) for lA in (0, 1) for lB in (0, 1)]
    cases += [dict(shared_b=True, gap=(8, 0, 16)), dict(lB=1, shared_a=True, gap=(0, 8, 32)), dict(offset=8), dict(offset=1)]
    for kw in cases:
        before = ab.adapt_launch_count()
        check_strided(M, N, K, batch, dtype, **kw)
        # (entries with a gap between them are copied only where TMA reads them in place anyway: else another route)
        assert "gap" in kw or ab.adapt_launch_count() - before <= 2, (shape, kw)
    check_strided(M, N, K, 3, dtype, gap=(3, 1, 7))


def integers(count, seed, dtype=ab.F16):
    return synth.draw_operand(1, count, ("integer", -4, 4), seed, dtype, "cuda").reshape(-1)


def expect_entries(A, sa, B, sb, C, sc, M, N, K, dtype, entries):
    for e in entries:
        _, want = og.gemm(synth.bits(A[e * sa:e * sa + M * K]), synth.bits(B[e * sb:e * sb + K * N]), M, N, K, dtype)
        assert np.array_equal(synth.bits(C[e * sc:e * sc + M * N]).reshape(want.shape), want), (M, N, K, e)


@pytest.mark.parametrize("offset", [0, 1])
@pytest.mark.parametrize("strides", [(8, 16), (64, 0), (16, 520), (40, 24), (3, 5)])
def test_strided_batch_of_entries_that_overlap_one_another(strides, offset):
    """Inputs closer together than an entry is long (sliding windows); read in place where rows and strides are 16-byte multiples."""
    init()
    M, N, K, batch, dt = 384, 512, 328, 120, ab.F16
    plan = ab.adapt_matmul_plan(M, N, K, dt)
    assert ab.adapt_plan_info(plan).family in (ab.FAM_UMMA_1CTA, ab.FAM_UMMA_2CTA)
    sa, sb = strides
    A, B = integers((batch - 1) * sa + M * K + offset, 5)[offset:], integers((batch - 1) * sb + K * N + offset, 6)[offset:]
    C = torch.full((batch * M * N,), float("nan"), dtype=torch.float16, device="cuda")
    st = torch.cuda.current_stream().cuda_stream
    before = ab.adapt_launch_count()
    ab.adapt_matmul_strided_batch(plan, A.data_ptr(), sa, B.data_ptr(), sb, C.data_ptr(), M * N, batch, st)
    launches = ab.adapt_launch_count() - before
    torch.cuda.synchronize()
    ab.adapt_poll_device_status(st)
    # in place: one launch; overlapping entries are not copied as a whole, so the others run one by one
    assert (launches == 1) == (offset == 0 and sa % 8 == 0 and sb % 8 == 0)
    expect_entries(A, sa, B, sb, C, M * N, M, N, K, dt, [0, 1, 37, 63, 64, batch - 1])


def test_copies_of_unaligned_entries_are_held_in_parts():
    """More copied bytes than are held at a time: several launches, a bounded workspace."""
    init()
    M, N, K, batch, dt = 370, 737, 98, 2000, ab.F16
    A, B = integers(batch * M * K, 7), integers(batch * K * N, 8)
    C = torch.full((batch * M * N,), float("nan"), dtype=torch.float16, device="cuda")
    stream = torch.cuda.Stream()
    plan = ab.adapt_matmul_plan(M, N, K, dt)
    torch.cuda.synchronize()
    before, free = ab.adapt_launch_count(), torch.cuda.mem_get_info()[0]
    ab.adapt_matmul_strided_batch(plan, A.data_ptr(), M * K, B.data_ptr(), K * N, C.data_ptr(), M * N, batch, stream.cuda_stream)
    torch.cuda.synchronize()
    ab.adapt_poll_device_status(stream.cuda_stream)
    copied = 2 * batch * (M * 112 + K * 752)                       # rows at a pitch of whole 32 bytes
    assert 4 <= 2 * -(-copied // (256 << 20)) == ab.adapt_launch_count() - before
    assert free - torch.cuda.mem_get_info()[0] <= 320 << 20        # 256 MB, an eighth more and the allocator's rounding
    expect_entries(A, M * K, B, K * N, C, M * N, M, N, K, dt, [0, 1, 1164, 1165, 1166, batch - 2, batch - 1])


def test_strided_batch_in_a_capture_on_a_stream_without_a_workspace():
    """The plan by itself needs no workspace, so the batch can be captured without a call before it; the copy of all entries, which
    would need one, is not an option there."""
    init()
    M, N, K, batch, dt = 100, 201, 130, 200, ab.F16
    plan = ab.adapt_matmul_plan(M, N, K, dt)
    assert ab.adapt_plan_info(plan).workspace_bytes == 0
    A, B = integers(batch * M * K, 9), integers(batch * K * N, 10)
    C = torch.full((batch * M * N,), float("nan"), dtype=torch.float16, device="cuda")
    args = (plan, A.data_ptr(), M * K, B.data_ptr(), K * N, C.data_ptr(), M * N, batch)
    before = ab.adapt_launch_count()
    ab.adapt_matmul_strided_batch(*args, torch.cuda.current_stream().cuda_stream)
    assert ab.adapt_launch_count() - before == 2                   # the copy and the tensor-core kernel
    C.fill_(float("nan"))
    side = torch.cuda.Stream()
    torch.cuda.synchronize()
    graph = torch.cuda.CUDAGraph()
    with torch.cuda.graph(graph, stream=side):
        ab.adapt_matmul_strided_batch(*args, side.cuda_stream)
    graph.replay()
    torch.cuda.synchronize()
    ab.adapt_poll_device_status(side.cuda_stream)
    expect_entries(A, M * K, B, K * N, C, M * N, M, N, K, dt, [0, 1, 99, batch - 1])
