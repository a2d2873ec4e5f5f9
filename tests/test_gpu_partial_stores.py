"""fp32 partials of plain tiles that leave through TMA boxes staged in the ring: exact on integers where boxes hang over the rows, the columns or
the k splits, for every tile and ring, and where a CTA has several units (only its last one's go that way)."""
import pytest
import torch

from paper_2608_10803_b200 import binding as ab
from paper_2608_10803_b200 import synth

from gpu_util import check_case, init

pytestmark = pytest.mark.gpu


@pytest.mark.parametrize("dtype", [ab.F16, ab.BF16])
@pytest.mark.parametrize("shape", [(65, 8, 2000), (72, 64, 1500), (97, 264, 1000), (129, 100, 1030), (160, 33, 3000), (257, 300, 700), (300, 2000, 640), (520, 4100, 400)])
def test_partials_of_every_plain_split(shape, dtype):
    M, N, K = shape
    init()
    A = synth.draw_operand(M, K, ("integer", -2, 2), 31, dtype, "cuda")
    B = synth.draw_operand(K, N, ("integer", -2, 2), 32, dtype, "cuda")
    seen = set()
    for lA, lB in [(0, 0), (1, 1)]:
        a = A if lA == 0 else A.t().contiguous()
        b = B if lB == 0 else B.t().contiguous()
        for c in ab.adapt_plan_candidates(M, N, K, dtype, lA, lB):
            plain = c.family in (ab.FAM_UMMA_1CTA, ab.FAM_UMMA_2CTA) and c.srcA != 3 and c.srcB != 3
            key = (c.family, c.BN, c.P_k, lA)
            if not plain or c.P_k < 2 or c.fused or key in seen or (c.P_k > 4 and c.P_k % 3):
                continue
            seen.add(key)
            check_case(M, N, K, dtype, a, b, lA, lB, plan=ab.adapt_matmul_plan_forced(M, N, K, dtype, lA, lB, c.tiling_key), exact=True)
    assert {ab.FAM_UMMA_1CTA, ab.FAM_UMMA_2CTA} <= {k[0] for k in seen} and len({k[1] for k in seen}) == 3
