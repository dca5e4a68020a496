"""sk_solve_precond at the edges of the fused pass over A: lanes per row (16 columns a lane: n = 16, 17, 32, 33,
64, 65, 128, 129, 256, 257, 512), row counts that leave warps and row groups partly empty, row strides, and rows
that are not 16-byte aligned (scalar loads). Bar as for the other shapes: the oracle's FP64 least-squares
solution to 1e-7 and a residual within 1e-8 of its own."""
import numpy as np
import pytest

import oracle
from paper_2606_20195_gb300 import inputs

pytestmark = pytest.mark.gpu


@pytest.mark.parametrize("m,n,pad,off", [
    (601, 1, 0, 0), (1000, 16, 0, 0), (1003, 17, 0, 0), (2048, 32, 0, 0), (2051, 33, 3, 0), (4099, 64, 0, 0),
    (4096, 64, 5, 0), (4097, 64, 8, 4), (5003, 64, 8, 1), (6007, 65, 0, 0), (8191, 128, 0, 0), (8193, 129, 0, 0),
    (9001, 256, 4, 0), (9005, 257, 0, 0), (12001, 512, 0, 0),
])
def test_precond_pass_edges(sk, dev, m, n, pad, off):
    import torch
    k = 4
    d = -(-4 * n // k) * k + 32
    A_h, b_h, _ = inputs.ls_problem_host(m, n, "incoherent", seed=m + n, noise=0.5)
    x_opt, r_opt = oracle.lstsq_tall(A_h, b_h)
    wide = torch.full((m, n + pad), float("nan"), device=dev)  # columns outside A must not be read into it
    A = wide[:, off:off + n]
    A.copy_(torch.from_numpy(A_h))
    plan = sk.Plan(d, m, k, 0, 3)
    x, _ = plan.solve_precond(A, torch.from_numpy(b_h).to(dev), tol=1e-12)
    xg = x.cpu().numpy()
    assert abs(oracle.residual_norm(A_h, b_h, xg) / r_opt - 1.0) <= 1e-8
    assert np.linalg.norm(xg - x_opt) <= 1e-7 * np.linalg.norm(x_opt)
    plan.close()
