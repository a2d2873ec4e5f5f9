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


def plans(M, N, K, dtype):
    """One forced plan of every kind, and the one the library picks."""
    out, seen = [ab.adapt_matmul_plan(M, N, K, dtype)], set()
    for c in ab.adapt_plan_candidates(M, N, K, dtype):
        key = (c.family, c.srcA, c.srcB, c.P_k > 1, c.fused, c.streamk, c.BN % 64 != 0, c.cluster > 1)
        if key not in seen:
            seen.add(key)
            out.append(ab.adapt_matmul_plan_forced(M, N, K, dtype, 0, 0, c.tiling_key))
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
