"""The panelled FP64 QR of sk_solve_sketched at the edges of its panels (4, 8 or 16 columns by n), with rows that
do not divide evenly over the CTAs, square sketches, several rows per thread, and columns that nearly depend on
earlier ones (where a panel is cut and its Gram matrix formed anew).

Reference: numpy's FP64 QR and least squares of the same matrix. x is returned in FP32 (6e-8 relative), and the
problems keep cond(A) 1e-16 and cond(A)^2 1e-16 ||residual|| / ||A x|| far below that: bar 1e-6 on x, and 1e-6 on
kappa = max |R_ii| / min |R_ii| (its FP64 error is of the order cond(A) 1e-16)."""
import numpy as np
import pytest

pytestmark = pytest.mark.gpu


def solve(sk, dev, W, n, rule=0, group=0):
    import torch
    d = W.shape[0]
    plan = sk.Plan(d, 4 * d, 1, rule, 1)
    if group:
        plan.set(sk.SK_PARAM_SOLVE_GROUP_ROWS, group)
    x = torch.empty(n, device=dev)
    sk.sk_solve_sketched(plan.handle, W, W.stride(0), n, x)
    st, kappa = plan.solve_status()
    x = x.cpu().numpy().astype(np.float64)
    plan.close()
    return st, kappa, x


def check(sk, dev, Wh, n, **kw):
    import torch
    st, kappa, x = solve(sk, dev, torch.from_numpy(Wh).to(dev), n, **kw)
    W = Wh.astype(np.float64)
    x_ref = np.linalg.lstsq(W[:, :n], W[:, n], rcond=None)[0]
    r = np.abs(np.diag(np.linalg.qr(W[:, :n], mode="r")))
    assert st == 0
    assert np.linalg.norm(x - x_ref) <= 1e-6 * np.linalg.norm(x_ref)
    assert abs(kappa / (r.max() / r.min()) - 1.0) <= 1e-6


@pytest.mark.parametrize("d,n", [
    (1, 1), (7, 1), (9, 3), (4, 4), (64, 4), (80, 5), (130, 8), (13, 13), (14, 14), (224, 14), (15, 15), (256, 16),
    (16, 16), (271, 17), (448, 28), (29, 29), (464, 29), (512, 32), (531, 33), (752, 47), (768, 48), (1024, 64),
    (1040, 65), (1600, 100), (2048, 128), (131, 131), (4096, 256), (40000, 16), (60001, 3), (1025, 511)])
def test_panel_edges(sk, dev, d, n):
    rng = np.random.default_rng(1000 * n + d)
    A = rng.standard_normal((d, n))
    if d == n:
        A += 4.0 * np.sqrt(n) * np.eye(n)
    b = A @ rng.standard_normal(n) + 1e-3 * rng.standard_normal(d)
    check(sk, dev, np.concatenate([A, b[:, None]], 1).astype(np.float32), n)


@pytest.mark.parametrize("d,n", [(512, 24), (1024, 64), (2048, 100)])
@pytest.mark.parametrize("eps", [1e-1, 1e-3, 1e-5])
def test_nearly_dependent_columns(sk, dev, d, n, eps):
    rng = np.random.default_rng(d + n)
    A = rng.standard_normal((d, n))
    for c in range(1, n, 3):  # every third column a small step away from its left neighbour
        A[:, c] = A[:, c - 1] + eps * rng.standard_normal(d)
    A *= 10.0 ** rng.uniform(-2, 2, n)  # column scales
    A = A.astype(np.float32)
    b = A.astype(np.float64) @ (rng.standard_normal(n) / np.linalg.norm(A.astype(np.float64), axis=0))
    b = b + 1e-6 * rng.standard_normal(d) * np.linalg.norm(b) / np.sqrt(d)
    # (column scales do not change the least-squares problem's difficulty, only x's: compare A x's columns)
    W = np.concatenate([A, b[:, None].astype(np.float32)], 1)
    import torch
    st, kappa, x = solve(sk, dev, torch.from_numpy(W).to(dev), n)
    W64 = W.astype(np.float64)
    s = np.linalg.norm(W64[:, :n], axis=0)
    y_ref = np.linalg.lstsq(W64[:, :n] / s, W64[:, n], rcond=None)[0]
    r = np.abs(np.diag(np.linalg.qr(W64[:, :n], mode="r")))
    assert st == 0
    assert np.linalg.norm(x * s - y_ref) <= 1e-6 * np.linalg.norm(y_ref)
    assert abs(kappa / (r.max() / r.min()) - 1.0) <= 1e-6


def test_zero_and_repeated_columns(sk, dev):
    import torch
    rng = np.random.default_rng(5)
    A = rng.standard_normal((300, 41)).astype(np.float32)
    A[:, 20] = 0.0  # an exactly zero column: a zero pivot
    st, _, x = solve(sk, dev, torch.from_numpy(A).to(dev), 40)
    assert st == sk.SK_ERR_NUMERIC and np.isnan(x).all()
    A[:, 20] = A[:, 3]  # a repeated column: a pivot of rounding size, as numpy's
    st, kappa, _ = solve(sk, dev, torch.from_numpy(A).to(dev), 40)
    assert st in (0, sk.SK_ERR_NUMERIC) and kappa >= 1e13


def test_tree_levels_and_types(sk, dev):
    import torch
    rng = np.random.default_rng(9)
    n = 21
    for rule, dt in ((1, torch.float16), (4, torch.bfloat16), (0, torch.float32)):
        W = torch.from_numpy(rng.standard_normal((900, n + 4)).astype(np.float32)).to(dt).to(dev)[:, :n + 1]
        W64 = W.cpu().double().numpy()
        x_ref = np.linalg.lstsq(W64[:, :n], W64[:, n], rcond=None)[0]
        for group in (0, 100):
            st, _, x = solve(sk, dev, W, n, rule, group)
            assert st == 0 and np.linalg.norm(x - x_ref) <= 1e-6 * np.linalg.norm(x_ref)
