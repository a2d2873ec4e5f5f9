"""Plans of tall pair tiles: calls whose buffers the tall tiles cannot serve run 256-row pair tiles, in one launch, also in lists and captures."""
import pytest
import torch

from paper_2608_10803_b200 import binding as ab
from paper_2608_10803_b200 import synth

from gpu_util import init

pytestmark = pytest.mark.gpu


@pytest.fixture(autouse=True)
def options():
    init()
    yield
    ab.adapt_set_option("shuffle_k", 0)


def stream():
    return torch.cuda.current_stream().cuda_stream


def integers(n, seed, dtype):
    return synth.draw_operand(1, n, ("integer", -3, 3), seed, dtype, "cuda").reshape(-1)


def product(A, B, M, N, K, lA, lB, rows):
    """The product's sampled rows: integers far below 2^53, exact in any order (and below 2^24, so one rounding follows)."""
    a = (A.view(K, M).t() if lA else A.view(M, K)).index_select(0, rows).double()
    return a @ (B.view(N, K).t() if lB else B.view(K, N)).double()


class Call:
    """Operands of one call, C (and D) a number of elements off an allocation's start."""

    def __init__(self, M, N, K, dtype, lA=0, lB=0, c_off=0, addmm=None, d_off=0):
        tall = next(c for c in ab.adapt_plan_candidates(M, N, K, dtype, lA, lB) if c.BM == 512)
        self.plan = ab.adapt_matmul_plan_forced(M, N, K, dtype, lA, lB, tall.tiling_key)
        self.A, self.B = integers(M * K, 1, dtype), integers(K * N, 2, dtype)
        self.flat = torch.full((M * N + 128,), float("nan"), dtype=self.A.dtype, device="cuda")
        self.at = 64 + c_off
        self.C = self.flat[self.at:self.at + M * N]
        self.vector = addmm == "bias"
        self.D = integers((N if self.vector else M * N) + d_off, 3, dtype)[d_off:] if addmm else None
        self.info = ab.adapt_plan_info_call(self.plan, self.C.data_ptr(), self.D.data_ptr() if addmm else 0, self.vector)
        self.rows = torch.unique(torch.tensor([0, 1, 127, 128, 255, 256, 257, 511, 512, M // 2, M - 257, M - 256, M - 2, M - 1], device="cuda").clamp(0, M - 1))
        want = product(self.A, self.B, M, N, K, lA, lB, self.rows)
        if addmm:
            want = 2.0 * want - (self.D if self.vector else self.D.view(M, N).index_select(0, self.rows)).double()
        self.want = want.to(self.A.dtype)
        self.shape = (M, N, K)

    def run(self, st):
        if self.D is None:
            ab.adapt_matmul(self.plan, self.A.data_ptr(), self.B.data_ptr(), self.C.data_ptr(), st)
        else:
            ab.adapt_addmm(self.plan, self.A.data_ptr(), self.B.data_ptr(), self.D.data_ptr(), self.vector, 2.0, -1.0, self.C.data_ptr(), st)

    def check(self):
        torch.cuda.synchronize()
        ab.adapt_poll_device_status(stream())
        M, N, K = self.shape
        assert torch.equal(self.C.view(M, N).index_select(0, self.rows), self.want), (self.shape, self.info.as_dict())
        assert torch.isfinite(self.C).all()
        assert torch.isnan(self.flat[:self.at]).all() and torch.isnan(self.flat[self.at + M * N:]).all(), "written outside C"


def launches(call, st):
    before = ab.adapt_launch_count()
    call.run(st)
    return ab.adapt_launch_count() - before


# in place, a short k range, over a copy, of row classes
SHAPES = [(1207, 4416, 2048), (5372, 4096, 896), (3623, 3616, 1219), (3367, 2608, 2955)]


def copies(call):
    return int(call.info.srcA == 1 or call.info.srcB == 1)


@pytest.mark.parametrize("shape", SHAPES)
@pytest.mark.parametrize("addmm", [None, "bias", "matrix"])
def test_unaligned_output(shape, addmm):
    for c_off in (8, 1):
        call = Call(*shape, ab.BF16, c_off=c_off, addmm=addmm)
        assert call.info.BM == 256 and launches(call, stream()) == 1 + copies(call)
        call.check()


@pytest.mark.parametrize("lA,lB", [(0, 0), (0, 1), (1, 0), (1, 1)])
def test_unaligned_or_short_added_matrix_and_reordered_k(lA, lB):
    for addmm, d_off, shape in [("bias", 1, (1208, 4416, 2048)), ("matrix", 4, (1208, 4416, 2048)), ("matrix", 0, (5376, 4096, 896))]:
        call = Call(*shape, ab.F16, lA, lB, addmm=addmm, d_off=d_off)
        assert call.info.BM == 256
        call.run(stream())
        call.check()
    call = Call(1208, 4416, 2048, ab.F16, lA, lB)
    assert call.info.BM == 512
    call.run(stream())
    call.check()
    ab.adapt_set_option("shuffle_k", 1)
    assert ab.adapt_plan_info_call(call.plan, call.C.data_ptr()).BM == 256
    call.run(stream())
    call.check()


def test_capture_and_lists():
    """No workspace that the plan does not need: such a call can be captured on any stream, and goes into a list as the plan's other calls do."""
    call = Call(1207, 4416, 2048, ab.BF16, c_off=8)
    side = torch.cuda.Stream()
    torch.cuda.synchronize()
    graph = torch.cuda.CUDAGraph()
    with torch.cuda.graph(graph, stream=side):
        assert launches(call, side.cuda_stream) == 1
    graph.replay()
    call.check()
    calls = [Call(*s, ab.BF16, c_off=o) for s in SHAPES for o in (8, 0)]
    ab.adapt_matmul_batch([c.plan for c in calls], [c.A.data_ptr() for c in calls], [c.B.data_ptr() for c in calls], [c.C.data_ptr() for c in calls], stream())
    for c in calls:
        c.check()
