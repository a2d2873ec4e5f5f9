"""The split-K reduction with the splits of an output shared by several threads: exact on integers around the split counts and
output sizes where the sharing starts and grows (8, 16, 32, 64, 128 splits; few and many outputs; ragged N), and with a fused add."""
import numpy as np
import pytest
import torch

from oracle import gemm as og
from paper_2608_10803_b200 import binding as ab
from paper_2608_10803_b200 import synth

from gpu_util import check_case, init

pytestmark = pytest.mark.gpu


@pytest.mark.parametrize("dtype", [ab.F16, ab.BF16])
@pytest.mark.parametrize("shape", [(1, 7, 20000), (37, 39, 26457), (64, 64, 16384), (130, 77, 9000), (16, 2048, 8192), (256, 256, 20000)])
def test_reduction_of_many_splits_exact(shape, dtype):
    M, N, K = shape
    init()
    st = torch.cuda.current_stream().cuda_stream
    A = synth.draw_operand(M, K, ("integer", -1, 1), 21, dtype, "cuda")       # |sums| stay exact in fp32
    B = synth.draw_operand(K, N, ("integer", -1, 1), 22, dtype, "cuda")
    D = synth.draw_operand(1, N, ("integer", -4, 4), 23, dtype, "cuda").reshape(-1)
    _, want = og.addmm_rows(synth.bits(A), synth.bits(B), synth.bits(D), M, N, K, dtype, 1.0, 2.0)
    seen = set()
    for c in ab.adapt_plan_candidates(M, N, K, dtype):
        if c.P_k < 7 or c.fused or c.P_k == c.cluster or c.P_k in seen:
            continue
        seen.add(c.P_k)
        plan = ab.adapt_matmul_plan_forced(M, N, K, dtype, 0, 0, c.tiling_key)
        check_case(M, N, K, dtype, A, B, plan=plan, exact=True)
        C = torch.full((M, N), float("nan"), dtype=A.dtype, device="cuda")
        ab.adapt_addmm(plan, A.data_ptr(), B.data_ptr(), D.data_ptr(), True, 1.0, 2.0, C.data_ptr(), st)
        torch.cuda.synchronize()
        assert np.array_equal(synth.bits(C).reshape(want.shape), want), (shape, c.P_k)
    assert seen and (max(seen) > 16 or K < 10000)
