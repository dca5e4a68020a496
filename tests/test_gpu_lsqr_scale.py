"""sk_solve_precond's iterates do not depend on the scale of b: multiplying b by a power of two multiplies x by it.
Everything but the scale of the step's coefficient alpha / ||u|| is then the same number, so solutions may differ
only by the order of the atomic sums, which the converged solution does not see above cond(A R^-1) times the
2^-48 of the float pairs u is kept in, over 30 iterations: bar 1e-12. Scales up to where the residuals' squares
still are FP64 numbers and A^T u FP32 ones."""
import numpy as np
import pytest

from paper_2606_20195_gb300 import inputs

pytestmark = pytest.mark.gpu


@pytest.mark.parametrize("n", [12, 40, 100])
def test_scale_of_b(sk, dev, n):
    import torch
    m, k = 3001, 4
    d = 8 * n
    A_h, b_h, _ = inputs.ls_problem_host(m, n, "incoherent", seed=n, noise=0.5)
    A = torch.from_numpy(A_h).to(dev)
    x = {}
    for e in (0, 60, 118, -60):
        b = torch.from_numpy(np.ldexp(b_h, e).astype(np.float32)).to(dev)
        plan = sk.Plan(d, m, k, 0, 3)
        y, _ = plan.solve_precond(A, b, tol=1e-14)
        x[e] = np.ldexp(y.cpu().numpy(), -e)
        plan.close()
    for e in (60, 118, -60):
        assert np.linalg.norm(x[e] - x[0]) <= 1e-12 * np.linalg.norm(x[0]), e
