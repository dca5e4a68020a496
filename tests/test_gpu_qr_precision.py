"""Digits of kappa = max |R_ii| / min |R_ii| where the columns share one direction: a panel's first column takes all
but a 1/900 of the squared norm out of the others. R's diagonal then depends on a difference that has to be formed
from the columns themselves and not from a Gram matrix of before.

Reference: Householder QR in long double. Bar: a squared norm may lose a factor of 16 (the panel's cut) of the
accuracy of a freshly formed one, which a sum of 1000 squares over some CTAs has to about 4 units of 2^-53; half
of that in the norm, and both the largest and the smallest diagonal entry count: 64 x 2^-53 = 7.1e-15."""
import numpy as np
import pytest

pytestmark = pytest.mark.gpu
BAR = 64 * 2.0 ** -53


def _kappa(W):
    A = W.astype(np.longdouble)
    n = A.shape[1]
    for j in range(n):
        x = A[j:, j]
        alpha = -np.copysign(np.sqrt((x * x).sum()), x[0])
        v = x.copy()
        v[0] -= alpha
        A[j:, j:] -= np.outer(v, (2 / (v * v).sum()) * (v @ A[j:, j:]))
        A[j, j] = alpha
    r = np.abs(np.diag(A))
    return r.max() / r.min()


@pytest.mark.parametrize("d,n", [(512, 29), (1024, 48)])
def test_kappa_of_columns_with_a_common_part(sk, dev, d, n):
    import torch
    worst = 0.0
    for seed in range(6):
        rng = np.random.default_rng(100 * n + seed)
        A = rng.standard_normal((d, 1)) * rng.choice([-1.0, 1.0], n) + rng.standard_normal((d, n)) / 30.0
        W = np.concatenate([A, rng.standard_normal((d, 1))], 1).astype(np.float32)
        plan = sk.Plan(d, 4 * d, 1, 0, 1)
        x = torch.empty(n, device=dev)
        sk.sk_solve_sketched(plan.handle, torch.from_numpy(W).to(dev), n + 1, n, x)
        st, kappa = plan.solve_status()
        assert st == 0
        worst = max(worst, abs(float(np.longdouble(kappa) / _kappa(W[:, :n]) - 1)))
        plan.close()
    assert worst <= BAR, worst
