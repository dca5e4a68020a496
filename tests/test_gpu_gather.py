"""Gather kernel (number 7 in SK_PARAM_LAST_KERNEL; AUTO from 65536 rows on, or 32768 unaligned ones): output
rows owned by half-warps, which fetch the rows of A that S sends to them. Small-integer data, so every chunk
total is exact and the result is bit-exact with the oracle's canonical order for every rule; random data within
the atomic-mode tolerance of the FP64 sketch (1e-5 FP32). The cases are the edges of the kernel's tiles (64
columns, 512 output rows in slots of 64, boxes of whole 1024 rows), short chunks (many items, partial boxes),
unaligned rows, 16-bit A, a row offset, lists so short that most rows take the overflow path, and a scratch
limit without room for chunk totals (another kernel then)."""
import numpy as np
import pytest

import oracle
from paper_2606_20195_gb300 import inputs

pytestmark = pytest.mark.gpu
GATHER = 7

SHAPES = [
    # m, n, row length, d, k, chunk rows, list capacity, row offset, type of A
    (65536, 64, 64, 4096, 1, 0, 0, 0, "float32"),
    (65551, 24, 28, 64, 1, 9000, 0, 0, "float32"),
    (65600, 128, 128, 2048, 2, 0, 0, 12345, "float32"),
    (65536, 64, 64, 4104, 4, 0, 0, 0, "float32"),
    (65536, 48, 48, 520, 1, 0, 8, 0, "float32"),
    (66000, 64, 72, 2056, 1, 0, 0, 0, "bfloat16"),
    (66000, 68, 72, 100, 1, 1000, 0, 99, "float16"),
    (32768, 17, 17, 528, 4, 0, 0, 0, "float32"),
    (40001, 33, 33, 1056, 4, 0, 0, 0, "float32"),
    (33000, 66, 67, 65, 1, 0, 16, 5, "float32"),
    (33000, 130, 131, 1539, 3, 0, 0, 0, "float32"),
]


def _sketch(sk, A, m, n, d, k, rule, dev, **params):
    import torch
    plan = sk.Plan(d, m, k, rule, 5, **params)
    Y = torch.full((d, n), 7.0, dtype=plan.out_dtype(), device=dev)
    for _ in range(2):  # the second call finds the chunk totals cleared
        plan.apply(A, Y)
    torch.cuda.synchronize()
    kern, R = plan.get(sk.SK_PARAM_LAST_KERNEL), plan.get(sk.SK_PARAM_LAST_CHUNK_ROWS)
    assert plan.get(sk.SK_PARAM_DEVICE_STATUS) == 0
    plan.close()
    return Y.cpu().numpy() if rule == 0 else Y.view(torch.int16).cpu().numpy().view(np.uint16), kern, R


@pytest.mark.parametrize("rule", [0, 1, 2, 3, 4])
@pytest.mark.parametrize("shape", SHAPES)
def test_gather_exact_on_integer_data(sk, dev, shape, rule):
    import torch
    m, n, lda, d, k, R, cap, off, a_type = shape
    A32 = np.zeros((m, lda), dtype=np.float32)
    A32[:, :n] = np.random.default_rng(m + n).integers(-3, 4, size=(m, n))
    A = torch.from_numpy(A32).to(dev).to(getattr(torch, a_type))[:, :n]
    params = {"list_cap": cap, "row_offset": off, **({"chunk_rows": R} if R else {})}
    got, kern, R_used = _sketch(sk, A, m, n, d, k, rule, dev, **params)
    assert kern == GATHER
    Af = np.zeros((off + m, n), dtype=np.float32)
    Af[off:] = A32[:, :n]
    ref = oracle.sketch_canonical(Af, d, k, 5, rule, R_used)
    assert np.array_equal(got, ref), np.count_nonzero(got != ref)


@pytest.mark.parametrize("shape", [(70001, 64, 2048, 1), (70001, 64, 4096, 4), (40001, 33, 1056, 4)])
def test_gather_random_within_tolerance(sk, dev, shape):
    import torch
    m, n, d, k = shape
    A = inputs.host_matrix(m, n, "incoherent", seed=21)
    got, kern, _ = _sketch(sk, torch.from_numpy(A).to(dev), m, n, d, k, 0, dev)
    assert kern == GATHER
    assert oracle.rel_fro(got.astype(np.float64), oracle.sketch_f64(A, d, k, 5)) <= 1e-5


def test_gather_infinities_stay_in_their_rows(sk, dev):
    import torch
    m, n, d, k = 65536, 64, 1024, 1
    A = np.random.default_rng(1).integers(-3, 4, size=(m, n)).astype(np.float32)
    A[17, 3], A[900, 40], A[901, 63] = np.inf, np.nan, -np.inf
    got, kern, R = _sketch(sk, torch.from_numpy(A).to(dev), m, n, d, k, 0, dev)
    assert kern == GATHER
    ref = oracle.sketch_canonical(A, d, k, 5, 0, R)
    assert np.array_equal(np.isfinite(got), np.isfinite(ref))
    assert np.array_equal(got[np.isfinite(ref)], ref[np.isfinite(ref)])


def test_gather_without_room_for_chunk_totals(sk, dev):
    import torch
    m, n, d, k = 65536, 128, 4096, 1  # (the tile kernel takes one slice per chunk here)
    A = np.random.default_rng(2).integers(-3, 4, size=(m, n)).astype(np.float32)
    got, kern, R = _sketch(sk, torch.from_numpy(A).to(dev), m, n, d, k, 1, dev, scratch_limit=64)
    assert kern == sk.SK_KERNEL_TILE
    assert np.array_equal(got, oracle.sketch_canonical(A, d, k, 5, 1, R))
