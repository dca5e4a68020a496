"""The workloads by which the speed of libsk is measured: what they are, their inputs, and their results in 64 bits.

Each case is one call of the library's public entry points (paper_2606_20195_gb300.sk) on inputs that are
already where a caller has them. `kind` says which call:

  apply    Y = S A of one matrix on the device (Plan.apply; 16-bit A goes through sk_apply_typed)
  host     the same from pinned host memory into host memory (sk_apply_host)
  batch    uneven matrices in one persistent launch (sk_batch_launch)
  solve    sketch-and-solve least squares (Plan.solve)
  precond  sketch-and-precondition least squares (Plan.solve_precond)

Sizes are those of the repository's benchmark, serving stream and tests, or lie between them.
"""
from __future__ import annotations

import math

import numpy as np
import torch

from paper_2606_20195_gb300 import sk

_DTYPES = {"float32": torch.float32, "float16": torch.float16, "bfloat16": torch.bfloat16}
_OUT = {"fp32": torch.float32, "bf16_rn": torch.bfloat16}  # the fp16 rules: float16
_RULES = ("fp32", "fp16_rn", "fp16_sr", "fp16_dither", "bf16_rn")


# ------------------------------------------------------------------------------------------ cases
def _apply(name, m, n, d, k, rule, a="float32", family="incoherent"):
    return {"name": name, "kind": "apply", "m": m, "n": n, "d": d, "k": k, "rule": rule, "a": a, "family": family}


def _solve(name, m, n, d, k, rule, family, kind="solve"):
    return {"name": name, "kind": kind, "m": m, "n": n, "d": d, "k": k, "rule": rule, "family": family}


def listed():
    return [
        # The smallest sketch of the configurations: launch and latency bound, called in a loop by users
        # with many small problems.
        _apply("small_k4_fp32", 16384, 16, 256, 4, "fp32"),
        # An odd number of rows and columns (no aligned rows, no TMA), stochastic rounding.
        _apply("ragged_k4_fp16_sr", 50001, 33, 1056, 4, "fp16_sr"),
        # The benchmark's headline: SparseStack of a tall matrix, FP16 accumulation.
        _apply("sweep_k8_fp16_rn", 1 << 22, 64, 4096, 8, "fp16_rn"),
        # The same with a bfloat16 matrix (half the bytes of A); first rows a scaled identity.
        _apply("sweep_k8_bf16_input", 1 << 22, 64, 4096, 8, "fp16_rn", "bfloat16", "coherent"),
        # CountSketch (one nonzero per column) of the same matrix in FP32.
        _apply("countsketch_n64_fp32", 1 << 22, 64, 4096, 1, "fp32"),
        # The paper's width (n = 1024) and SparseStack's usual four nonzeros, dithered rounding.
        _apply("wide_k4_fp16_dither", 1 << 19, 1024, 2048, 4, "fp16_dither"),
        # A caller whose matrix is in host memory: CountSketch at the paper's width, copies included.
        {"name": "host_countsketch_n1024", "kind": "host", "m": 1 << 17, "n": 1024, "d": 2048, "k": 1,
         "rule": "fp16_rn", "family": "incoherent"},
        # Many matrices of uneven size in one launch, as a service sketches the requests of one step.
        {"name": "batch_48_uneven_k4", "kind": "batch", "count": 48, "lo": 12.0, "hi": 20.0, "shapes": 5, "k": 4,
         "rule": "fp16_rn"},
        # One least-squares request of a service: latency from the sketch to x.
        _solve("solve_serving_n64", 1 << 16, 64, 1024, 4, "fp16_rn", "incoherent"),
        # Sketch-and-solve of a tall coherent problem.
        _solve("solve_tall_n128", 1 << 23, 128, 2048, 8, "fp16_sr", "coherent"),
        # The paper's least-squares experiment (coherent, rows permuted): 1024 columns, FP64 QR of 4096 rows.
        _solve("solve_paper_n1024", 1 << 19, 1024, 4096, 4, "fp32", "permuted"),
        # Least squares to full accuracy: the sketch's R as a preconditioner for LSQR on A.
        _solve("precond_n128", 1 << 21, 128, 2048, 8, "fp32", "coherent", "precond"),
    ]


def _log(rng, lo, hi):
    return int(round(2.0 ** rng.uniform(math.log2(lo), math.log2(hi))))


def draw(rng):
    kind = rng.choice(("apply", "apply", "apply", "apply", "solve", "solve", "batch", "precond", "host"))
    if kind == "batch":
        return {"kind": kind, "count": rng.randint(8, 48), "lo": 12.0, "hi": rng.uniform(15.0, 20.0),
                "shapes": rng.randrange(1 << 20), "k": 4, "rule": rng.choice(_RULES)}
    if kind in ("solve", "precond"):
        n = rng.choice((16, 32, 48, 64, 100, 128, 200, 256))
        k = 8 if kind == "precond" else rng.choice((1, 4, 8))
        d = 16 * n
        m = min(_log(rng, max(1 << 14, 2 * d), 1 << 21) + rng.choice((0, 0, 1, 13)), (1 << 28) // n)
        # (CountSketch collides the identity rows of a coherent matrix: not a problem users solve with it)
        family = "incoherent" if k == 1 else rng.choice(("incoherent", "coherent"))
        return {"kind": kind, "m": m, "n": n, "d": d, "k": k, "rule": "fp32" if kind == "precond" else
                rng.choice(_RULES[:4]), "family": family}
    k = rng.choice((1, 1, 2, 4, 4, 8, 8))
    n = _log(rng, 4, 1024)
    if rng.random() < 0.75:
        n = max(4, n // 4 * 4)  # aligned rows
    ratio = rng.choice((2, 4, 8, 16, 32, 64))
    d = max(8, min(ratio * n, 16384) // 8 * 8)
    limit = (1 << 28 if n % 8 == 0 else 1 << 24) // (16 if kind == "host" else 1)
    m = _log(rng, 1 << 10, max(1 << 11, min(1 << 22, limit // n))) + rng.choice((0, 0, 0, 1, 7))
    c = {"kind": kind, "m": m, "n": n, "d": d, "k": k, "rule": rng.choice(_RULES),
         "family": rng.choice(("incoherent", "incoherent", "coherent", "adversarial"))}
    if kind == "apply":
        c["a"] = rng.choice(("float32", "float32", "float32", "float16", "bfloat16"))
    return c


def _shapes(case):
    """(m, n, d, family) of a batch: m log-uniform, n from the benchmark's widths, d = 32 n, every other matrix coherent."""
    r = np.random.default_rng(case["shapes"])
    out = []
    for i in range(case["count"]):
        m = int(2.0 ** r.uniform(case["lo"], case["hi"]))
        n = int(r.choice((8, 16, 32, 64, 128)))
        out.append((m, n, 32 * n, "incoherent" if i % 2 == 0 else "coherent"))
    return out


# ------------------------------------------------------------------------------------------ inputs
def _generator(seed):
    g = torch.Generator(device="cuda")
    g.manual_seed(int(seed))
    return g


def _matrix(g, m, n, family):
    if family == "adversarial":  # one entry per row
        A = torch.zeros((m, n), device="cuda")
        r = torch.arange(m, device="cuda")
        A[r, r % n] = torch.randn(m, generator=g, device="cuda")
        return A
    A = torch.randn((m, n), generator=g, device="cuda")
    if family == "coherent":  # a scaled identity on top of small noise
        A.mul_(1e-3)
        q = min(m, n)
        A[:q] = 0.0
        A.diagonal().fill_(1e3)
    return A


def _problem(case, seed):
    """(A, b) of a least-squares case."""
    g = _generator(seed)
    m, n, family = case["m"], case["n"], case["family"]
    if family == "permuted":  # identity rows and a small Gaussian tail, rows permuted
        G = torch.randn((m - n, n), generator=g, device="cuda").mul_(1e-3 / math.sqrt(m - n))
        xs = torch.randn(n, generator=g, device="cuda")
        A = torch.cat([torch.eye(n, device="cuda"), G])
        b = torch.cat([xs + 0.5 * torch.randn(n, generator=g, device="cuda"), G @ xs])
        del G
        p = torch.randperm(m, generator=g, device="cuda")
        return A[p].contiguous(), b[p].contiguous()
    A = _matrix(g, m, n, family)
    xs = torch.randn(n, generator=g, device="cuda")
    noise = 1e-6 if family == "coherent" else 0.1
    return A, A @ xs + noise * torch.randn(m, generator=g, device="cuda")


def _inputs(case, seed):
    if case["kind"] in ("solve", "precond"):
        return _problem(case, seed)
    if case["kind"] == "batch":
        g = _generator(seed)
        return [_matrix(g, m, n, family) for m, n, _, family in _shapes(case)]
    return _matrix(_generator(seed), case["m"], case["n"], case["family"]).to(_DTYPES[case.get("a", "float32")])


class _Batch:
    """A batch handle and the tensors it points to."""

    def __init__(self, items, rule):
        self.items = items
        self.handle = sk.sk_batch_create(items, rule)

    def __del__(self):
        sk.sk_batch_destroy(self.handle)


def prepare(case, seed):
    kind, data = case["kind"], _inputs(case, seed)
    state = {"kind": kind}
    if kind == "batch":
        dt = _OUT.get(case["rule"], torch.float16)
        items = [{"A": A, "Y": torch.empty((d, n), dtype=dt, device="cuda"), "m": m, "n": n, "d": d, "k": case["k"],
                  "seed": seed + i} for i, (A, (m, n, d, _)) in enumerate(zip(data, _shapes(case)))]
        state["batch"] = _Batch(items, sk.RULES[case["rule"]])
        return state
    plan = state["plan"] = sk.Plan(case["d"], case["m"], case["k"], case["rule"], seed=seed)
    if kind in ("solve", "precond"):
        state["A"], state["b"] = data
        state["x"] = torch.empty(case["n"], dtype=torch.float32 if kind == "solve" else torch.float64, device="cuda")
    elif kind == "host":
        state["A"] = torch.empty(data.shape, dtype=data.dtype, pin_memory=True)
        state["A"].copy_(data)
        state["Y"] = torch.empty((case["d"], case["n"]), dtype=plan.out_dtype(), pin_memory=True)
    else:
        state["A"] = data
        state["Y"] = torch.empty((case["d"], case["n"]), dtype=plan.out_dtype(), device="cuda")
    return state


def run(state):
    kind = state["kind"]
    if kind == "batch":
        b = state["batch"]
        sk.sk_batch_launch(b.handle)
        return [it["Y"] for it in b.items]
    plan = state["plan"]
    if kind == "apply":
        return plan.apply(state["A"], state["Y"])
    if kind == "host":
        A, Y = state["A"], state["Y"]
        sk.sk_apply_host(plan.handle, A.data_ptr(), A.stride(0), A.shape[1], Y.data_ptr())
        return Y
    if kind == "solve":
        return plan.solve(state["A"], state["b"], state["x"])
    x, _ = plan.solve_precond(state["A"], state["b"], state["x"])
    return x


# ------------------------------------------------------------------------------------------ work
def work(case):
    """Bytes: the matrix (and b) read once, the result written once. Operations: one addition per element
    of A and nonzero of its column of S; for the solves also the Householder QR of the sketch, and for the
    preconditioned one ten products with A and its transpose."""
    kind, k = case["kind"], case["k"]
    es_y = 4 if case["rule"] == "fp32" else 2
    if kind == "batch":
        s = _shapes(case)
        return {"bytes": sum(4 * m * n + es_y * d * n for m, n, d, _ in s), "flops": sum(k * m * n for m, n, _, _ in s)}
    m, n, d = case["m"], case["n"], case["d"]
    if kind in ("solve", "precond"):
        flops = k * m * (n + 1) + 2 * n * n * (d - n / 3)
        if kind == "precond":
            flops += 10 * 4 * m * n
        return {"bytes": 4 * m * (n + 1) + 4 * n, "flops": flops}
    es_a = 4 if case.get("a", "float32") == "float32" else 2
    return {"bytes": es_a * m * n + es_y * d * n, "flops": k * m * n}


# ------------------------------------------------------------------------------------------ results in 64 bits
def _i64(v):
    return v - (1 << 64) if v >= 1 << 63 else v


def _shr(z, s):
    return (z >> s) & ((1 << (64 - s)) - 1)


def _pattern(i0, i1, j, d, k, seed):
    """(target row, sign) of rows i0..i1-1 in block j of S: SplitMix64 output i * ceil(k/2) + j/2 + 1 from the
    seed, high half for even j, multiply-shift into the block, sign from the lowest bit."""
    kp, B = (k + 1) // 2, d // k
    idx = torch.arange(i0, i1, device="cuda", dtype=torch.int64) * kp + (j // 2 + 1)
    z = idx * _i64(0x9E3779B97F4A7C15) + int(seed)
    z = (z ^ _shr(z, 30)) * _i64(0xBF58476D1CE4E5B9)
    z = (z ^ _shr(z, 27)) * _i64(0x94D049BB133111EB)
    z = z ^ _shr(z, 31)
    w = z & 0xFFFFFFFF if j % 2 else _shr(z, 32)
    return j * B + ((w * B) >> 32), 1.0 - 2.0 * (w & 1).double()


def _sketch64(A, d, k, seed):
    m, n = A.shape
    Y = torch.zeros((d, n), dtype=torch.float64, device="cuda")
    step = max(1, (1 << 27) // n)
    for i0 in range(0, m, step):
        i1 = min(m, i0 + step)
        a = A[i0:i1].double()
        for j in range(k):
            t, s = _pattern(i0, i1, j, d, k, seed)
            Y.index_add_(0, t, a * s[:, None])
    return Y / math.sqrt(k)


def _least_squares64(M, b):
    """argmin ||M x - b|| by normal equations, refined twice (well-conditioned M, rows in chunks)."""
    m, n = M.shape
    step = max(n, (1 << 26) // n)
    G = torch.zeros((n, n), dtype=torch.float64, device="cuda")
    for i0 in range(0, m, step):
        a = M[i0:i0 + step].double()
        G += a.T @ a
    L = torch.linalg.cholesky(G)
    x = torch.zeros(n, dtype=torch.float64, device="cuda")
    for _ in range(4):
        g = torch.zeros(n, dtype=torch.float64, device="cuda")
        for i0 in range(0, m, step):
            a = M[i0:i0 + step].double()
            g += a.T @ (b[i0:i0 + step].double() - a @ x)
        x = x + torch.cholesky_solve(g[:, None], L)[:, 0]
    return x


def exact(case, seed):
    data, k = _inputs(case, seed), case["k"]
    if case["kind"] == "batch":
        return [_sketch64(A, d, k, seed + i) for i, (A, (_, _, d, _)) in enumerate(zip(data, _shapes(case)))]
    if case["kind"] == "solve":
        A, b = data
        return _least_squares64(_sketch64(A, case["d"], k, seed), _sketch64(b[:, None], case["d"], k, seed)[:, 0])
    if case["kind"] == "precond":
        return _least_squares64(*data)
    return _sketch64(data, case["d"], k, seed)
