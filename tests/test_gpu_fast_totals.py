"""Sketches that AUTO finishes in one launch (short slices of each chunk; past a grid barrier the same kernel adds
the chunk totals into Y): the launch count and the scratch show that this form ran, and one plan serves matrices of
different width and height in turn, growing and shrinking, with data whose chunk totals cancel to subnormal
numbers of either sign in between (an FP32 reduction leaves -0 there). Integer data, so every chunk total is
exact and the result is bit-exact with the oracle's canonical order."""
import numpy as np
import pytest

import oracle

pytestmark = pytest.mark.gpu
BARRIER = 256  # bytes of barrier words in front of the chunk totals


def _bits(Y, rule):
    import torch
    return Y.cpu().numpy() if rule == 0 else Y.view(torch.int16).cpu().numpy().view(np.uint16)


def _ints(m, n, seed):
    return np.random.default_rng(seed).integers(-3, 4, size=(m, n)).astype(np.float32)


@pytest.mark.parametrize("shape", [(16384, 16, 256, 4), (5001, 33, 48, 4), (9000, 20, 64, 1), (4097, 1, 256, 4),
                                   (8000, 64, 8192, 4), (3000, 12, 4096, 2), (200, 5, 16, 1)])
@pytest.mark.parametrize("rule", [0, 2])
def test_one_launch(sk, dev, shape, rule):
    import torch
    m, n, d, k = shape
    A = _ints(m, n, m + n)
    plan = sk.Plan(d, m, k, rule, 11)
    Y = torch.full((d, n), 7.0, dtype=plan.out_dtype(), device=dev)
    for _ in range(2):  # the second call finds barrier words and totals cleared
        plan.apply(torch.from_numpy(A).to(dev), Y)
    torch.cuda.synchronize()
    R = plan.get(sk.SK_PARAM_LAST_CHUNK_ROWS)
    assert plan.get(sk.SK_PARAM_LAST_LAUNCHES) == 1 and plan.get(sk.SK_PARAM_LAST_KERNEL) == sk.SK_KERNEL_TILE
    assert plan.get(sk.SK_PARAM_SCRATCH_BYTES) == 4 + BARRIER + 4 * -(-m // R) * d * n
    assert plan.get(sk.SK_PARAM_DEVICE_STATUS) == 0
    assert np.array_equal(_bits(Y, rule), oracle.sketch_canonical(A, d, k, 11, rule, R))
    plan.close()


def test_one_plan_many_widths(sk, dev):
    import torch
    d, k, rule = 256, 4, 0
    plan = sk.Plan(d, 16384, k, rule, 11)
    rng = np.random.default_rng(2)
    for i, (m, n) in enumerate([(16384, 16), (9000, 12), (16384, 16), (4096, 20), (16384, 24), (5000, 4), (12000, 20)]):
        plan.set(sk.SK_PARAM_ROWS, m)
        # neighbouring rows cancel to a few units of 2^-136: totals that end as subnormals or signed zeros
        tiny = np.repeat(1.0 + rng.integers(0, 8, (m // 2, n)) * 2.0 ** -10, 2, axis=0) * 2.0 ** -126
        tiny[1::2] *= -1.0
        tiny = np.ascontiguousarray(tiny + (rng.integers(0, 3, tiny.shape) - 1) * 2.0 ** -136).astype(np.float32)
        Y = torch.empty((d, n), device=dev)
        plan.apply(torch.from_numpy(tiny).to(dev), Y)
        A = _ints(m, n, i)
        plan.apply(torch.from_numpy(A).to(dev), Y)
        torch.cuda.synchronize()
        assert plan.get(sk.SK_PARAM_LAST_LAUNCHES) == 1
        assert np.array_equal(Y.cpu().numpy(), oracle.sketch_canonical(A, d, k, 11, rule, plan.get(sk.SK_PARAM_LAST_CHUNK_ROWS)))
    assert plan.get(sk.SK_PARAM_DEVICE_STATUS) == 0
    plan.close()


@pytest.mark.parametrize("shape", [(16384, 16, 256, 4), (5001, 33, 48, 4), (4097, 1, 256, 4)])
def test_call_after_a_barrier_gave_up(sk, dev, shape):
    # A barrier wait of one cycle runs out; the next call on the plan must find its scratch clean.
    import torch
    m, n, d, k = shape
    A = _ints(m, n, 3)
    plan = sk.Plan(d, m, k, 1, 11, sketch_wait_cycles=1)
    Ad, Y = torch.from_numpy(A).to(dev), torch.empty((d, n), dtype=torch.float16, device=dev)
    for _ in range(3):
        plan.apply(Ad, Y)
    assert plan.get(sk.SK_PARAM_DEVICE_STATUS) == 1
    plan.set(sk.SK_PARAM_SKETCH_WAIT_CYCLES, 0)
    plan.set(sk.SK_PARAM_SOLVE_WAIT_CYCLES, 1)  # (the QR's own bound)
    for _ in range(2):
        plan.apply(Ad, Y)
        torch.cuda.synchronize()
        assert plan.get(sk.SK_PARAM_LAST_LAUNCHES) == 1
        assert np.array_equal(_bits(Y, 1), oracle.sketch_canonical(A, d, k, 11, 1, plan.get(sk.SK_PARAM_LAST_CHUNK_ROWS)))
    plan.close()


@pytest.mark.parametrize("shape", [(16384, 16, 256, 4), (33000, 33, 1056, 4)])
def test_graph_outlives_the_plans_scratch(sk, dev, shape):
    # A graph captured after an eager call replays after a larger call has made the plan's scratch grow.
    import torch
    m, n, d, k = shape
    A, B = _ints(m, n, 1), _ints(m, 4 * n, 2)
    Ad, Bd = torch.from_numpy(A).to(dev), torch.from_numpy(B).to(dev)
    plan = sk.Plan(d, m, k, 1, 11)
    Y = torch.empty((d, n), dtype=torch.float16, device=dev)
    Z = torch.empty((d, 4 * n), dtype=torch.float16, device=dev)
    plan.apply(Ad, Y)
    torch.cuda.synchronize()
    graph = torch.cuda.CUDAGraph()
    with torch.cuda.graph(graph):
        plan.apply(Ad, Y)
    plan.apply(Bd, Z)
    torch.cuda.synchronize()
    for _ in range(2):
        Y.zero_()
        graph.replay()
        plan.apply(Bd, Z)
        torch.cuda.synchronize()
        R = plan.get(sk.SK_PARAM_LAST_CHUNK_ROWS)
        assert np.array_equal(_bits(Y, 1), oracle.sketch_canonical(A, d, k, 11, 1, R))
        assert np.array_equal(_bits(Z, 1), oracle.sketch_canonical(B, d, k, 11, 1, R))
    assert plan.get(sk.SK_PARAM_DEVICE_STATUS) == 0
    plan.close()


@pytest.mark.parametrize("shape", [(16384, 16, 256, 4), (33000, 33, 1056, 4), (8000, 64, 8192, 4)])
def test_one_plan_on_several_streams(sk, dev, shape):
    # Nothing orders the streams' calls, and each has its own A and Y. (Sketches that need no chunk totals; those of
    # the register kernel for FP32 A, say, always share the plan's.)
    import torch
    m, n, d, k = shape
    plan = sk.Plan(d, m, k, 1, 11)
    streams = [torch.cuda.Stream() for _ in range(4)]
    A = [_ints(m, n, s) for s in range(4)]
    Ad = [torch.from_numpy(a).to(dev) for a in A]
    Y = [[torch.empty((d, n), dtype=torch.float16, device=dev) for _ in range(8)] for _ in range(4)]
    plan.apply(Ad[0], Y[0][0])
    torch.cuda.synchronize()
    for i in range(8):
        for s in range(4):
            plan.apply(Ad[s], Y[s][i], streams[s])
    torch.cuda.synchronize()
    assert plan.get(sk.SK_PARAM_DEVICE_STATUS) == 0
    R = plan.get(sk.SK_PARAM_LAST_CHUNK_ROWS)
    for s in range(4):
        ref = oracle.sketch_canonical(A[s], d, k, 11, 1, R)
        for i in range(8):
            assert np.array_equal(_bits(Y[s][i], 1), ref), (s, i)
    plan.close()


@pytest.mark.parametrize("before", [64, 2000])  # rows of an earlier call: too few for totals, and some
def test_eager_call_beside_another_streams_capture(sk, dev, before):
    # The scratch of an eager call is allocated, or grown, while another stream is being captured (global mode).
    import torch
    m, n, d, k = 16384, 16, 256, 4
    A = _ints(m, n, 1)
    Ad = torch.from_numpy(A).to(dev)
    first, plan = sk.Plan(d, m, k, 1, 11), sk.Plan(d, m, k, 1, 11)
    Y, Z = (torch.zeros((d, n), dtype=torch.float16, device=dev) for _ in range(2))
    side = torch.cuda.Stream()
    first.apply(Ad, Z)
    small = torch.from_numpy(A[:before]).to(dev)
    plan.set(sk.SK_PARAM_ROWS, before)
    plan.apply(small, Y)  # (the plan's status word)
    plan.set(sk.SK_PARAM_ROWS, m)
    torch.cuda.synchronize()
    graph = torch.cuda.CUDAGraph()
    with torch.cuda.graph(graph):
        first.apply(Ad, Z)
        plan.apply(Ad, Y, side)
    torch.cuda.synchronize()
    ref = oracle.sketch_canonical(A, d, k, 11, 1, plan.get(sk.SK_PARAM_LAST_CHUNK_ROWS))
    assert np.array_equal(_bits(Y, 1), ref)
    Z.zero_()
    graph.replay()
    torch.cuda.synchronize()
    assert np.array_equal(_bits(Z, 1), ref)
    first.close()
    plan.close()


@pytest.mark.parametrize("R", [1, 7, 300])
@pytest.mark.parametrize("a_type,k", [("float32", 1), ("bfloat16", 4)])
def test_short_chunks(sk, dev, R, a_type, k):
    import torch
    m, n, d = 65536, 20 if a_type == "float32" else 64, 640
    A = _ints(m, n, R)
    plan = sk.Plan(d, m, k, 0, 11, chunk_rows=R)
    Y = plan.apply(torch.from_numpy(A).to(dev).to(getattr(torch, a_type)))
    torch.cuda.synchronize()
    assert plan.get(sk.SK_PARAM_LAST_KERNEL) == sk.SK_KERNEL_TILE
    assert plan.get(sk.SK_PARAM_SCRATCH_BYTES) <= 4 + BARRIER + 4 * m * n
    # (k = 1 has scale 1 and integer sums, and k = 4 sums of halves: exact in any order)
    assert np.array_equal(_bits(Y, 0), oracle.sketch_canonical(A, d, k, 11, 0, R))
    plan.close()


def test_apply_then_solve_under_the_solves_limit(sk, dev):
    import torch
    m, n, d, k = 16384, 16, 256, 4
    A = _ints(m, n, 5)
    Ad, Y = torch.from_numpy(A).to(dev), torch.empty((d, n), device=dev)
    b = torch.from_numpy(A @ np.arange(1.0, n + 1, dtype=np.float32)).to(dev)
    alone, plan = sk.Plan(d, m, k, 0, 11), sk.Plan(d, m, k, 0, 11)
    sk.sk_solve_sketched(alone.handle, torch.zeros((d, n + 1), device=dev), n + 1, n, torch.empty(n, device=dev))
    plan.apply(Ad, Y)
    plan.set(sk.SK_PARAM_SCRATCH_LIMIT, alone.get(sk.SK_PARAM_SCRATCH_BYTES) + 4)
    x = plan.solve(Ad, b)  # A x = b holds exactly, so the sketched solution is 1 .. n
    assert plan.solve_status()[0] == 0
    assert np.allclose(x.cpu().numpy(), np.arange(1, n + 1), rtol=1e-5)
    plan.apply(Ad, Y)
    torch.cuda.synchronize()
    assert np.array_equal(_bits(Y, 0), oracle.sketch_canonical(A, d, k, 11, 0, plan.get(sk.SK_PARAM_LAST_CHUNK_ROWS)))
    alone.close()
    plan.close()
