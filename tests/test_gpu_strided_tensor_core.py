"""Strided batches on the tensor-core kernel: one launch (and at most one copy) for all entries, bit-exact on integers."""
import pytest

from paper_2608_10803_b200 import binding as ab

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
