"""AddMM where the GEMM kernel itself adds D: every kind of output path (TMA boxes, halo tiles, thread stores, fused split-K, stream-K,
warp-level, CUDA-core and one-launch tiles) with aligned and unaligned D, matrix and bias, bit-exact on integers, and in place."""
import numpy as np
import pytest
import torch

from oracle import gemm as og
from paper_2608_10803_b200 import binding as ab
from paper_2608_10803_b200 import synth

from gpu_util import init

pytestmark = pytest.mark.gpu


def plans(M, N, K, dtype, lA=0, lB=0):
    """One forced plan of every kind, and the one the library picks."""
    out, seen = [ab.adapt_matmul_plan(M, N, K, dtype, lA, lB)], set()
    for c in ab.adapt_plan_candidates(M, N, K, dtype, lA, lB):
        key = (c.family, c.srcA, c.srcB, c.P_k > 1, c.fused, c.streamk, c.BN % 64 != 0, c.cluster > 1)
        if key not in seen:
            seen.add(key)
            out.append(ab.adapt_matmul_plan_forced(M, N, K, dtype, lA, lB, c.tiling_key))
    return out


@pytest.mark.parametrize("dtype", [ab.F16, ab.BF16])
@pytest.mark.parametrize("shape", [(129, 320, 96), (300, 1001, 64), (257, 200, 130), (33, 4100, 200), (5, 640, 600), (700, 1, 65), (1, 700, 64), (40, 50, 20),
                                   (2560, 1024, 2048)])
def test_addmm_exact_on_every_output_path(shape, dtype):
    M, N, K = shape
    init()
    st = torch.cuda.current_stream().cuda_stream
    A = synth.position_coded(M, K, dtype, 7, "cuda")
    B = synth.position_coded(K, N, dtype, 5, "cuda").contiguous()
    flat = synth.draw_operand(1, M * N + 8, ("integer", -8, 8), 43, dtype, "cuda").reshape(-1)
    rows = np.arange(M) if M * N * K <= 1 << 27 else np.array([0, 1, 127, 128, 129, 255, 256, M // 2, M - 2, M - 1])
    idx = torch.from_numpy(rows).cuda()
    for vector in (False, True):
        for offset in (0, 1, 8):
            D = flat[offset:offset + (N if vector else M * N)]
            Dh = synth.bits(D)
            _, want = og.addmm_rows(synth.bits(A), synth.bits(B), Dh, M, N, K, dtype, 2.0, -3.0, rows=rows)
            for plan in plans(M, N, K, dtype):
                C = torch.full((M, N), float("nan"), dtype=A.dtype, device="cuda")
                ab.adapt_addmm(plan, A.data_ptr(), B.data_ptr(), D.data_ptr(), vector, 2.0, -3.0, C.data_ptr(), st)
                torch.cuda.synchronize()
                ab.adapt_poll_device_status(st)
                info = ab.adapt_plan_info(plan)
                tag = (shape, vector, offset, ab.FAMILY_NAMES[info.family], info.BN, info.P_k, info.fused, info.streamk)
                assert np.array_equal(synth.bits(C.index_select(0, idx)).reshape(want.shape), want), tag
                if not vector and offset != 1:
                    inplace = flat.clone()[offset:offset + M * N]
                    ab.adapt_addmm(plan, A.data_ptr(), B.data_ptr(), inplace.data_ptr(), False, 2.0, -3.0, inplace.data_ptr(), st)
                    torch.cuda.synchronize()
                    assert torch.equal(inplace.view(torch.int16), C.reshape(-1).view(torch.int16)), ("in place",) + tag


def same_values(got, want):
    """Bit for bit, any NaN for any NaN (16-bit patterns of the same type)."""
    got, want = got.reshape(-1).astype(np.uint16), want.reshape(-1).astype(np.uint16)
    exponent = 0x7C00 if same_values.dtype == ab.F16 else 0x7F80
    nan = lambda x: ((x & exponent) == exponent) & ((x & (0x7FFF - exponent)) != 0)
    return bool((nan(got) == nan(want)).all() and (got == want)[~nan(want)].all())


@pytest.mark.parametrize("dtype", [ab.F16, ab.BF16])
@pytest.mark.parametrize("layouts", [(0, 1), (1, 0), (1, 1)])
@pytest.mark.parametrize("shape", [(129, 320, 96), (300, 1001, 64), (257, 200, 130), (33, 2100, 200), (5, 640, 600), (700, 1, 65), (40, 50, 20)])
def test_addmm_exact_in_the_other_layouts(shape, layouts, dtype):
    M, N, K = shape
    init()
    st = torch.cuda.current_stream().cuda_stream
    A, B, D = (synth.draw_operand(1, n, ("integer", -4, 4), seed, dtype, "cuda").reshape(-1) for n, seed in ((M * K, 51), (K * N, 52), (M * N, 53)))
    for vector in (False, True):
        d = D[:N] if vector else D
        _, want = og.addmm_rows(synth.bits(A), synth.bits(B), synth.bits(d), M, N, K, dtype, 0.5, 3.0, *layouts)
        for plan in plans(M, N, K, dtype, *layouts):
            C = torch.full((M, N), float("nan"), dtype=A.dtype, device="cuda")
            ab.adapt_addmm(plan, A.data_ptr(), B.data_ptr(), d.data_ptr(), vector, 0.5, 3.0, C.data_ptr(), st)
            torch.cuda.synchronize()
            ab.adapt_poll_device_status(st)
            info = ab.adapt_plan_info(plan)
            assert np.array_equal(synth.bits(C).reshape(want.shape), want), (shape, layouts, vector, ab.FAMILY_NAMES[info.family], info.BN, info.P_k, info.fused)


@pytest.mark.parametrize("dtype", [ab.F16, ab.BF16])
@pytest.mark.parametrize("shape", [(129, 320, 96), (300, 201, 64), (65, 200, 130), (33, 1100, 200), (5, 640, 600), (40, 50, 20)])
def test_addmm_of_infinities_nan_and_the_types_largest_values(shape, dtype):
    """Special values of A, B and D reach exactly the outputs that the arithmetic gives; with beta = 0 a finite D adds nothing."""
    M, N, K = shape
    init()
    same_values.dtype = dtype
    st = torch.cuda.current_stream().cuda_stream
    A, B, D = (synth.draw_operand(r, c, ("integer", 1, 4), seed, dtype, "cuda") for r, c, seed in ((M, K, 61), (K, N, 62), (M, N, 63)))
    big = torch.finfo(A.dtype).max
    D[0, 0], D[M - 1, N - 1], D[M // 2, N // 2], D[1, N - 2], D[2, 3] = float("inf"), float("-inf"), float("nan"), -big, big
    E = D.clone()
    A[3, K - 1], B[K - 1, N - 3], A[4, 0] = float("inf"), float("-inf"), float("nan")
    with np.errstate(all="ignore"):
        cases = [(d, *ab_, og.addmm_rows(synth.bits(A), synth.bits(B), synth.bits(d), M, N, K, dtype, *ab_)[1]) for d in (D, E[M // 2]) for ab_ in ((1.0, 1.0), (-2.0, 0.5))]
    for d, alpha, beta, want in cases:
        for plan in plans(M, N, K, dtype):
            C = torch.full((M, N), 7.0, dtype=A.dtype, device="cuda")
            ab.adapt_addmm(plan, A.data_ptr(), B.data_ptr(), d.data_ptr(), d.dim() == 1, alpha, beta, C.data_ptr(), st)
            torch.cuda.synchronize()
            ab.adapt_poll_device_status(st)
            info = ab.adapt_plan_info(plan)
            assert same_values(synth.bits(C), want), (shape, alpha, ab.FAMILY_NAMES[info.family], info.BN, info.P_k, info.fused)
    finite = torch.full((M, N), big, dtype=A.dtype, device="cuda")
    for plan in plans(M, N, K, dtype):
        plain, zero = (torch.full((M, N), 7.0, dtype=A.dtype, device="cuda") for _ in range(2))
        ab.adapt_matmul(plan, A.data_ptr(), B.data_ptr(), plain.data_ptr(), st)
        ab.adapt_addmm(plan, A.data_ptr(), B.data_ptr(), finite.data_ptr(), False, 1.0, 0.0, zero.data_ptr(), st)
        torch.cuda.synchronize()
        assert same_values(synth.bits(zero), synth.bits(plain))


@pytest.mark.parametrize("vector", [False, True])
def test_small_output_goes_through_the_sums_or_not_with_the_same_result(vector):
    """One row of tiles that its threads store (rows of C off 32-byte boundaries): two launches over the workspace, and in a capture on a
    stream without one, where it must not grow, the kernel adds D itself."""
    M, N, K, dtype = 128, 5608, 256, ab.F16
    init()
    plan = ab.adapt_matmul_plan(M, N, K, dtype)
    info = ab.adapt_plan_info(plan)
    assert info.family in (ab.FAM_UMMA_1CTA, ab.FAM_UMMA_2CTA) and info.P_k == 1 and info.workspace_bytes == 0
    A, B, D = (synth.draw_operand(1, n, ("integer", -4, 4), seed, dtype, "cuda").reshape(-1) for n, seed in ((M * K, 71), (K * N, 72), (M * N, 73)))
    d = D[:N] if vector else D
    _, want = og.addmm_rows(synth.bits(A), synth.bits(B), synth.bits(d), M, N, K, dtype, 0.5, 3.0)
    C = torch.full((M, N), float("nan"), dtype=A.dtype, device="cuda")
    args = (plan, A.data_ptr(), B.data_ptr(), d.data_ptr(), vector, 0.5, 3.0, C.data_ptr())
    before = ab.adapt_launch_count()
    ab.adapt_addmm(*args, torch.cuda.current_stream().cuda_stream)
    assert ab.adapt_launch_count() - before == 2
    torch.cuda.synchronize()
    assert np.array_equal(synth.bits(C).reshape(want.shape), want)
    C.fill_(float("nan"))
    side = torch.cuda.Stream()
    torch.cuda.synchronize()
    graph, before = torch.cuda.CUDAGraph(), ab.adapt_launch_count()
    with torch.cuda.graph(graph, stream=side):
        ab.adapt_addmm(*args, side.cuda_stream)
    assert ab.adapt_launch_count() - before == 1
    graph.replay()
    torch.cuda.synchronize()
    ab.adapt_poll_device_status(side.cuda_stream)
    assert np.array_equal(synth.bits(C).reshape(want.shape), want)
