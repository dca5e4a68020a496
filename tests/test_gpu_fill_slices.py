"""Short work-item slices (chunks split until the items fill the GPU): small-integer data, where every chunk
total is exact, so the result is bit-exact with the oracle's canonical order however the chunk is split.
Row counts around the 64-row minimum of a slice, ragged last chunks, a row offset, unaligned rows, one
column, and a scratch limit that leaves no room for chunk totals (one slice per chunk then)."""
import numpy as np
import pytest

import oracle

pytestmark = pytest.mark.gpu

SHAPES = [
    # m, n, d, k, chunk rows, row offset
    (16384, 16, 256, 4, 0, 0),
    (5001, 33, 1056, 4, 0, 0),
    (127, 5, 16, 1, 0, 0),
    (64, 4, 8, 2, 0, 0),
    (9000, 64, 1024, 4, 4096, 100),
    (4097, 1, 256, 4, 0, 0),
    (3000, 12, 65536, 2, 0, 7),
]


def _run(sk, A, d, k, rule, seed, dev, **params):
    import torch
    plan = sk.Plan(d, A.shape[0], k, rule, seed, **params)
    Y = torch.full((d, A.shape[1]), 7.0, dtype=plan.out_dtype(), device=dev)
    for _ in range(2):  # the second call finds the chunk totals cleared
        plan.apply(torch.from_numpy(A).to(dev), Y)
    torch.cuda.synchronize()
    R, launches = plan.get(sk.SK_PARAM_LAST_CHUNK_ROWS), plan.get(sk.SK_PARAM_LAST_LAUNCHES)
    assert plan.get(sk.SK_PARAM_DEVICE_STATUS) == 0
    plan.close()
    return Y.cpu().numpy() if rule == 0 else Y.view(torch.int16).cpu().numpy().view(np.uint16), R, launches


@pytest.mark.parametrize("rule", [0, 1, 2, 4])
@pytest.mark.parametrize("shape", SHAPES)
def test_filled_slices_exact_on_integer_data(sk, dev, rule, shape):
    m, n, d, k, R, off = shape
    A = np.random.default_rng(m + n).integers(-3, 4, size=(m, n)).astype(np.float32)
    got, R_used, _ = _run(sk, A, d, k, rule, 11, dev, row_offset=off, **({"chunk_rows": R} if R else {}))
    Af = np.zeros((off + m, n), dtype=np.float32)
    Af[off:] = A
    ref = oracle.sketch_canonical(Af, d, k, 11, rule, R_used)
    assert np.array_equal(got, ref), np.count_nonzero(got != ref)


def test_no_room_for_chunk_totals(sk, dev):
    m, n, d, k = 16384, 16, 256, 4
    A = np.random.default_rng(0).integers(-3, 4, size=(m, n)).astype(np.float32)
    full, R, l2 = _run(sk, A, d, k, 1, 3, dev)
    tight, _, l1 = _run(sk, A, d, k, 1, 3, dev, scratch_limit=64)
    assert (l1, l2) == (1, 1)
    ref = oracle.sketch_canonical(A, d, k, 3, 1, R)
    assert np.array_equal(full, ref) and np.array_equal(tight, ref)
