"""Lists whose launches run on several streams: calls that depend on one another across streams, in groups and alone, and a list captured on a
stream that has never been used."""
import random

import pytest
import torch

from paper_2608_10803_b200 import binding as ab
from paper_2608_10803_b200 import synth

from gpu_util import init

pytestmark = pytest.mark.gpu


def stream():
    return torch.cuda.current_stream().cuda_stream


def mixed_list(r, count):
    """Calls over a few shared buffers: (plan, A, B, C) as (tensor, first element) with big calls (launched by themselves) and small ones
    (grouped) reading and overwriting one another's rows."""
    n, dt = 768, ab.F16
    pool = [synth.draw_operand(n, n, synth.U11, 900 + i, dt, "cuda") / 32 for i in range(7)]
    weights = [synth.draw_operand(n, n, synth.U11, 950 + i, dt, "cuda") / 16 for i in range(3)]
    big, rows, thin = ab.adapt_matmul_plan(n, n, n, dt), ab.adapt_matmul_plan(64, n, 64, dt), ab.adapt_matmul_plan(64, 64, n, dt)
    split = ab.adapt_matmul_plan(32, 32, 16 * n, dt)               # k splits: a workspace
    calls = []
    for _ in range(count):
        src, dst = r.sample(range(len(pool)), 2)
        at = 64 * n * r.randrange(n // 64)
        kind = r.choice(["big", "big", "rows", "rows", "thin", "split"])
        if kind == "big":
            calls.append((big, (pool[src], 0), (weights[r.randrange(3)], 0), (pool[dst], 0)))
        elif kind == "rows":                                           # the first 64 x 64 elements of a row block times 64 x n of a weight
            calls.append((rows, (pool[src], at), (weights[r.randrange(3)], 64 * n * r.randrange(n // 64)), (pool[dst], 64 * n * r.randrange(n // 64))))
        elif kind == "thin":
            calls.append((thin, (pool[src], at), (weights[r.randrange(3)], 0), (pool[dst], 64 * n * r.randrange(n // 64))))
        else:
            calls.append((split, (pool[src], 0), (weights[r.randrange(3)], 0), (pool[dst], at)))
    return pool, calls


def pointers(calls):
    return [[c[j][0].data_ptr() + 2 * c[j][1] for c in calls] for j in (1, 2, 3)]


@pytest.mark.parametrize("streams", [1, 2, 4])
@pytest.mark.parametrize("seed", range(6))
def test_dependent_calls_on_several_streams_keep_their_order(seed, streams):
    init()
    pool, calls = mixed_list(random.Random(seed), 60)
    plans, (A, B, C) = [c[0] for c in calls], pointers(calls)
    families = {ab.adapt_plan_info(p).family for p in plans}
    assert ab.FAM_CLUSTER in families and families & {ab.FAM_UMMA_1CTA, ab.FAM_UMMA_2CTA} and any(ab.adapt_plan_info(p).workspace_bytes for p in plans)
    start = [x.clone() for x in pool]
    for p, a, b, c in zip(plans, A, B, C):
        ab.adapt_matmul(p, a, b, c, stream())
    torch.cuda.synchronize()
    want = [x.clone() for x in pool]
    assert sum(not torch.equal(x, y) for x, y in zip(want, start)) >= 5
    ab.adapt_set_option("batch_streams", streams)
    try:
        for _ in range(5):
            for x, y in zip(pool, start):
                x.copy_(y)
            ab.adapt_matmul_batch(plans, A, B, C, stream())
            got = [x.clone() for x in pool]                            # after the join, on the caller's stream
            torch.cuda.synchronize()
            ab.adapt_poll_device_status(stream())
            for x, y in zip(got, want):
                assert torch.equal(x.view(torch.int16), y.view(torch.int16))
    finally:
        ab.adapt_set_option("batch_streams", 4)


def test_list_that_has_run_can_be_captured_on_another_stream():
    """Its workspaces belong to the library's streams, not to the one it first ran on."""
    init()
    pool, calls = mixed_list(random.Random(11), 40)
    plans, (A, B, C) = [c[0] for c in calls], pointers(calls)
    start = [x.clone() for x in pool]
    ab.adapt_matmul_batch(plans, A, B, C, stream())
    torch.cuda.synchronize()
    want = [x.clone() for x in pool]
    for x, y in zip(pool, start):
        x.copy_(y)
    args = [ab.pointer_array(x) for x in (plans, A, B, C)]
    side = torch.cuda.Stream()
    torch.cuda.synchronize()
    graph = torch.cuda.CUDAGraph()
    with torch.cuda.graph(graph, stream=side):
        ab.adapt_matmul_batch(*args, side.cuda_stream)
    graph.replay()
    torch.cuda.synchronize()
    ab.adapt_poll_device_status(stream())
    for x, y in zip(pool, want):
        assert torch.equal(x.view(torch.int16), y.view(torch.int16))
