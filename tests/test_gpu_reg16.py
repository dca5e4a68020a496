"""Register kernel on 16-bit A (AUTO at k >= 2, n >= 32, blocks of at most 512 rows): 64-column tiles, 512
output rows per work item. Small-integer data, so every chunk total is exact and the result is bit-exact
with the oracle's canonical order; the cases are tile edges (n around 32, 64 and 128, d around 512), lists
that overflow (list capacity 1), a row offset and a row stride, and a scratch limit without room for chunk
totals (the tile kernel then)."""
import numpy as np
import pytest

import oracle

pytestmark = pytest.mark.gpu

SHAPES = [
    # m, n, padded row length, d, k, chunk rows, list capacity, row offset
    (20011, 64, 64, 4096, 8, 4096, 0, 0),
    (9000, 65, 72, 1024, 2, 2048, 0, 0),
    (9000, 33, 40, 520, 4, 2048, 0, 0),
    (7000, 130, 136, 504, 8, 0, 0, 0),
    (20000, 64, 64, 2048, 8, 8192, 1, 0),
    (5000, 32, 80, 96, 3, 1000, 0, 7777),
]


def _sketch(sk, A, m, n, d, k, rule, dev, **params):
    import torch
    plan = sk.Plan(d, m, k, rule, 5, **params)
    Y = torch.full((d, n), 7.0, dtype=plan.out_dtype(), device=dev)
    plan.apply(A, Y)
    torch.cuda.synchronize()
    kern, R = plan.get(sk.SK_PARAM_LAST_KERNEL), plan.get(sk.SK_PARAM_LAST_CHUNK_ROWS)
    assert plan.get(sk.SK_PARAM_DEVICE_STATUS) == 0
    plan.close()
    return Y.cpu().numpy() if rule == 0 else Y.view(torch.int16).cpu().numpy().view(np.uint16), kern, R


@pytest.mark.parametrize("a_type", ["float16", "bfloat16"])
@pytest.mark.parametrize("rule", [0, 1, 2, 4])
@pytest.mark.parametrize("shape", SHAPES)
def test_reg16_exact_on_integer_data(sk, dev, shape, rule, a_type):
    import torch
    m, n, lda, d, k, R, cap, off = shape
    A32 = np.zeros((m, lda), dtype=np.float32)
    A32[:, :n] = np.random.default_rng(m + n).integers(-3, 4, size=(m, n))
    A = torch.from_numpy(A32).to(dev).to(getattr(torch, a_type))[:, :n]
    params = {"list_cap": cap, "row_offset": off, **({"chunk_rows": R} if R else {})}
    got, kern, R_used = _sketch(sk, A, m, n, d, k, rule, dev, **params)
    assert kern == sk.SK_KERNEL_REGISTER
    Af = np.zeros((off + m, n), dtype=np.float32)
    Af[off:] = A32[:, :n]
    ref = oracle.sketch_canonical(Af, d, k, 5, rule, R_used)
    assert np.array_equal(got, ref), np.count_nonzero(got != ref)


def test_reg16_infinities_stay_in_their_rows(sk, dev):
    # An infinity, a NaN and the largest bfloat16 reach only the output rows that S sends them to.
    import torch
    m, n, d, k = 4000, 64, 1024, 4
    A32 = np.random.default_rng(1).integers(-3, 4, size=(m, n)).astype(np.float32)
    A32[17, 3], A32[900, 40], A32[901, 63] = np.inf, np.nan, 3.3895314e38
    A = torch.from_numpy(A32).to(dev).bfloat16()
    got, kern, _ = _sketch(sk, A, m, n, d, k, 0, dev)
    assert kern == sk.SK_KERNEL_REGISTER
    ref = oracle.sketch_canonical(A.float().cpu().numpy(), d, k, 5, 0, 4096)
    assert np.array_equal(np.isfinite(got), np.isfinite(ref))
    assert np.array_equal(got[np.isfinite(ref)], ref[np.isfinite(ref)])


def test_reg16_without_room_for_chunk_totals(sk, dev):
    import torch
    m, n, d, k = 4000, 64, 512, 4
    A32 = np.random.default_rng(2).integers(-3, 4, size=(m, n)).astype(np.float32)
    A = torch.from_numpy(A32).to(dev).half()
    got, kern, R = _sketch(sk, A, m, n, d, k, 1, dev, scratch_limit=64)
    assert kern == sk.SK_KERNEL_TILE
    assert np.array_equal(got, oracle.sketch_canonical(A32, d, k, 5, 1, R))
