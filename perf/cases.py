"""The timed workloads of this library: what its users have it do, through the public entry points.

Five operators: ``matmul`` (adapt_matmul), ``addmm`` (adapt_addmm), ``step`` (one linear layer's training step: forward with
bias and both gradients, which are the same calls on column-major views of the operands), ``strided`` (adapt_matmul_strided_batch)
and ``group`` (adapt_matmul_batch).  Shapes are those of ``synth.py``'s workloads (the recommendation layers, the LLM layers, the
large and tall-K products, the paper-named ragged shape, the log-uniform sweep) or of the same ranges.
"""
from __future__ import annotations

import math
import random

import torch

from paper_2608_10803_b200 import binding as ab
from paper_2608_10803_b200 import synth

MAC_LIMIT = 2 ** 38            # of one product, as in the sweep
ELEMENT_LIMIT = 6 * 10 ** 8    # of A, B and C together


def _matmul(M, N, K, dtype, layoutA=0, layoutB=0, **more):
    return dict(op="matmul", M=M, N=N, K=K, dtype=dtype, layoutA=layoutA, layoutB=layoutB, **more)


def listed():
    return [
        # the smallest calls: a 256^3 product, and a batch of 64 requests through a recommendation layer (launch latency)
        _matmul(256, 256, 256, "f16", name="square 256"),
        _matmul(64, 1024, 1024, "f16", name="reco layer, 64 rows"),
        # the same layer with its bias, at a batch of 1000
        dict(op="addmm", M=1000, N=1024, K=1024, dtype="f16", layoutB=0, bias=True, alpha=1.0, beta=1.0, name="reco layer + bias, 1000 rows"),
        # LLM layers: decode (16 tokens stream the weights once) and prefill (2048 tokens)
        _matmul(16, 14336, 4096, "bf16", name="decode, 16 tokens"),
        _matmul(2048, 14336, 4096, "bf16", name="prefill, 2048 tokens"),
        # one linear layer's training step: forward with bias, gradient of the input, gradient of the weights
        dict(op="step", M=2048, N=4096, K=4096, dtype="bf16", name="training step, 2048 tokens"),
        # attention scores: one small product per head, Q row-major, K's rows as the columns
        dict(op="strided", batch=96, M=128, N=128, K=64, dtype="bf16", layoutB=1, shared_b=False, name="96 heads 128x128x64"),
        # the list of small layers of different shapes that a recommendation model issues together
        dict(op="group", count=48, shape_seed=42, lo=16, hi=1024, dtype="f16", name="group of 48 layers"),
        # a skewed product whose rows are not 16-byte multiples (the paper's ablation shape)
        _matmul(12288, 688, 16991, "f16", name="ragged 12288x688x16991"),
        # an output that outweighs its operands, rows of odd length
        _matmul(20000, 20001, 12, "bf16", name="wide output 20000x20001x12"),
        # a contraction over a long K into a small tile (weight gradients over many tokens)
        _matmul(256, 256, 262144, "bf16", name="tall K 256x256x262144"),
        # the largest: compute-bound
        _matmul(8192, 8192, 8192, "bf16", name="square 8192"),
    ]


def _log(rng, lo, hi):
    return max(lo, min(hi, int(math.exp(rng.uniform(math.log(lo), math.log(hi + 1))))))


def _fits(M, N, K, macs=MAC_LIMIT):
    return 2 ** 22 <= M * N * K <= macs and M * K + K * N + M * N <= ELEMENT_LIMIT


def _shape(rng, macs=MAC_LIMIT):
    """M, N, K of one product: sweep-like, a recommendation layer, an LLM layer or a long contraction."""
    while True:
        kind = rng.choice(["sweep", "sweep", "reco", "llm", "tall"])
        if kind == "sweep":
            M, N, K = (_log(rng, 1, 100000) for _ in range(3))
        elif kind == "reco":
            M, N, K = _log(rng, 1, 100000), _log(rng, 128, 2048), _log(rng, 128, 2048)
            if rng.random() < 0.5:
                N, K = (N + 63) // 64 * 64, (K + 63) // 64 * 64
        elif kind == "llm":
            M, N, K = _log(rng, 1, 8192), _log(rng, 1024, 16384) // 64 * 64, _log(rng, 1024, 16384) // 64 * 64
        else:
            M, N, K = _log(rng, 16, 512), _log(rng, 16, 512), _log(rng, 16384, 262144)
        if _fits(M, N, K, macs):
            return M, N, K


def draw(rng):
    dtype = rng.choice(["f16", "bf16"])
    op = rng.choice(["matmul", "matmul", "matmul", "matmul", "addmm", "addmm", "step", "strided", "group"])
    if op == "matmul":
        M, N, K = _shape(rng)
        return _matmul(M, N, K, dtype, layoutA=int(rng.random() < 0.125), layoutB=int(rng.random() < 0.25))
    if op == "addmm":
        M, N, K = _shape(rng)
        return dict(op="addmm", M=M, N=N, K=K, dtype=dtype, layoutB=int(rng.random() < 0.25), bias=rng.random() < 0.6,
                    alpha=rng.choice([1.0, 0.5]), beta=rng.choice([1.0, -2.0]))
    if op == "step":
        while True:
            M, N, K = _log(rng, 64, 8192), _log(rng, 128, 8192), _log(rng, 128, 8192)
            if rng.random() < 0.7:
                N, K = (N + 15) // 16 * 16, (K + 15) // 16 * 16
            if _fits(M, N, K, 2 ** 36):
                return dict(op="step", M=M, N=N, K=K, dtype=dtype)
    if op == "strided":
        while True:
            batch, M, N, K = _log(rng, 2, 256), _log(rng, 8, 1024), _log(rng, 8, 1024), _log(rng, 8, 1024)
            if rng.random() < 0.5:
                N, K = (N + 15) // 16 * 16, (K + 15) // 16 * 16
            if 2 ** 22 <= batch * M * N * K <= 2 ** 35:
                return dict(op="strided", batch=batch, M=M, N=N, K=K, dtype=dtype, layoutB=int(rng.random() < 0.5), shared_b=rng.random() < 0.25)
    return dict(op="group", count=rng.randint(8, 64), shape_seed=rng.randrange(1 << 30), lo=rng.choice([1, 8, 16]), hi=_log(rng, 256, 2048), dtype=dtype)


def _dtype(case):
    return ab.F16 if case["dtype"] == "f16" else ab.BF16


def _group_shapes(case):
    r = random.Random(case["shape_seed"])
    return [tuple(_log(r, case["lo"], case["hi"]) for _ in range(3)) for _ in range(case["count"])]


class _Draw:
    """Operands of one case, each from a seed of its own."""

    def __init__(self, case, seed):
        self.dtype, self.seed = _dtype(case), 1_000_003 * (int(seed) + 1)

    def __call__(self, rows, cols, dist):
        self.seed += 1
        return synth.draw_operand(rows, cols, dist, self.seed, self.dtype, "cuda")

    def activations(self, rows, cols):
        return self(rows, cols, synth.U11)

    def weights(self, rows, cols, fan_in):
        return self(rows, cols, ("normal", 0.0, 1.0 / math.sqrt(fan_in)))

    def empty(self, rows, cols):
        return torch.empty((rows, cols), dtype=synth.torch_dtype(self.dtype), device="cuda")


def prepare(case, seed):
    ab.adapt_init(0)
    d, dt = _Draw(case, seed), _dtype(case)
    s = {"op": case["op"], "stream": torch.cuda.current_stream().cuda_stream}
    if case["op"] == "group":
        shapes = _group_shapes(case)
        s["A"] = [d.activations(M, K) for M, N, K in shapes]
        s["B"] = [d.weights(K, N, K) for M, N, K in shapes]
        s["C"] = [d.empty(M, N) for M, N, K in shapes]
        plans = ab.adapt_plan_many([(M, N, K, dt) for M, N, K in shapes])
        s["args"] = [ab.pointer_array(plans)] + [ab.pointer_array([t.data_ptr() for t in s[k]]) for k in "ABC"]
        return s
    M, N, K = case["M"], case["N"], case["K"]
    la, lb = case.get("layoutA", 0), case.get("layoutB", 0)
    if case["op"] == "strided":
        b = case["batch"]
        nb = 1 if case["shared_b"] else b
        s["A"], s["C"], s["batch"] = d.activations(b * M, K), d.empty(b * M, N), b
        s["B"] = d.activations(nb * N, K) if lb else d.activations(nb * K, N)
        s["strides"] = (M * K, 0 if case["shared_b"] else K * N, M * N)
        s["plan"] = ab.adapt_matmul_plan(M, N, K, dt, 0, lb)
        return s
    s["A"] = d.activations(K, M) if la else d.activations(M, K)
    s["B"] = d.weights(N, K, K) if lb else d.weights(K, N, K)
    s["C"] = d.empty(M, N)
    s["plan"] = ab.adapt_matmul_plan(M, N, K, dt, la, lb)
    if case["op"] == "addmm":
        s["bias"], s["alpha"], s["beta"] = case["bias"], case["alpha"], case["beta"]
        s["D"] = d.activations(1, N) if case["bias"] else d.activations(M, N)
    elif case["op"] == "step":
        # forward X[M,K] W[K,N] + b; gradient of the input dX = dY W^T (W's storage read column-major as N x K); gradient of
        # the weights dW = X^T dY (X's storage read column-major as K x M)
        s["D"], s["dY"] = d.activations(1, N), d.activations(M, N)
        s["dX"], s["dW"] = d.empty(M, K), d.empty(K, N)
        s["plan_dX"] = ab.adapt_matmul_plan(M, K, N, dt, ab.ROW_MAJOR, ab.COL_MAJOR)
        s["plan_dW"] = ab.adapt_matmul_plan(K, N, M, dt, ab.COL_MAJOR, ab.ROW_MAJOR)
    return s


def run(s):
    op = s["op"]
    if op == "group":
        ab.adapt_matmul_batch(*s["args"], s["stream"])
        return s["C"]
    A, B, C = s["A"].data_ptr(), s["B"].data_ptr(), s["C"].data_ptr()
    if op == "matmul":
        ab.adapt_matmul(s["plan"], A, B, C, s["stream"])
    elif op == "addmm":
        ab.adapt_addmm(s["plan"], A, B, s["D"].data_ptr(), s["bias"], s["alpha"], s["beta"], C, s["stream"])
    elif op == "strided":
        sa, sb, sc = s["strides"]
        ab.adapt_matmul_strided_batch(s["plan"], A, sa, B, sb, C, sc, s["batch"], s["stream"])
    else:
        dY = s["dY"].data_ptr()
        ab.adapt_addmm(s["plan"], A, B, s["D"].data_ptr(), True, 1.0, 1.0, C, s["stream"])
        ab.adapt_matmul(s["plan_dX"], dY, B, s["dX"].data_ptr(), s["stream"])
        ab.adapt_matmul(s["plan_dW"], A, dY, s["dW"].data_ptr(), s["stream"])
        return {"Y": s["C"], "dX": s["dX"], "dW": s["dW"]}
    return s["C"]


def work(case):
    if case["op"] == "group":
        shapes = _group_shapes(case)
        return {"bytes": sum(2.0 * (M * K + K * N + M * N) for M, N, K in shapes), "flops": sum(2.0 * M * N * K for M, N, K in shapes)}
    M, N, K = case["M"], case["N"], case["K"]
    if case["op"] == "strided":
        b = case["batch"]
        return {"bytes": 2.0 * (b * M * K + (1 if case["shared_b"] else b) * K * N + b * M * N), "flops": 2.0 * b * M * N * K}
    if case["op"] == "step":       # X, W, dY read once each, Y, dX, dW written once each, and the bias
        return {"bytes": 2.0 * (2 * M * K + 2 * K * N + 2 * M * N + N), "flops": 6.0 * M * N * K}
    extra = (N if case["bias"] else M * N) if case["op"] == "addmm" else 0
    return {"bytes": 2.0 * (M * K + K * N + M * N + extra), "flops": 2.0 * M * N * K}


def tolerance(case):
    # Against the same product in 64 bits a result shows the rounding of its 16-bit output: 2.1e-4 (fp16) and 1.66e-3 (bf16) in
    # the 2-norm, 4.9e-4 and 3.9e-3 of the value at most, whatever the operator and K (12 to 262144).  Four times that.
    return {"rel": 8e-4, "max": 2e-3} if case["dtype"] == "f16" else {"rel": 6.6e-3, "max": 1.6e-2}
