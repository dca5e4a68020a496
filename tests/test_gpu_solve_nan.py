"""kappa of sk_solve_status is at least 1 whatever the sketch holds: a NaN in the first column makes all of R NaN,
an infinity its first diagonal entry infinite."""
import math

import numpy as np
import pytest

pytestmark = pytest.mark.gpu


@pytest.mark.parametrize("n", [1, 5, 40, 300])
@pytest.mark.parametrize("bad", [float("nan"), float("inf")])
def test_kappa_without_a_finite_diagonal(sk, dev, n, bad):
    import torch
    d = 2 * n + 7
    W = np.random.default_rng(n).standard_normal((d, n + 1)).astype(np.float32)
    W[d // 2, 0] = bad
    plan = sk.Plan(d, 4 * d, 1, 0, 1)
    x = torch.empty(n, device=dev)
    sk.sk_solve_sketched(plan.handle, torch.from_numpy(W).to(dev), n + 1, n, x)
    st, kappa = plan.solve_status()
    assert st == 0 and math.isinf(kappa) and kappa > 0
    plan.close()
