"""FP64 passes over A (two rows a warp) at odd row counts and widths, and the FP64 residual of single
solves, against FP64 products on the host: [f; g] = [b - r - A x; -A^T r] to n u and sqrt(m) u times the
sums of magnitudes.
"""
import numpy as np
import pytest
import torch

from conftest import dev

pytestmark = pytest.mark.gpu

U = 2.0 ** -53


@pytest.mark.parametrize("m,n", [(1, 1), (3, 2), (15, 3), (16, 4), (17, 16), (31, 31), (2431, 33), (2433, 64), (4865, 187),
                                 (5000, 188), (3001, 256), (2999, 500), (2500, 513), (1217, 1000), (1300, 1023)])
def test_residual(lsq, handle, m, n):
    g = np.random.default_rng(m + n)
    A, b, x, r = (g.standard_normal(k) for k in ((m, n), m, n, m))
    f, gg = (torch.zeros(k, dtype=torch.float64, device="cuda") for k in (m, n))
    lsq.lsq_residual(handle, dev(A), dev(b), m, n, "f64", None, dev(x), dev(r), f, gg)
    aA = np.abs(A)
    assert np.all(np.abs(f.cpu().numpy() - (b - r - A @ x)) <= 2 * (n + 3) * U * (np.abs(b) + np.abs(r) + aA @ np.abs(x)))
    assert np.all(np.abs(gg.cpu().numpy() + A.T @ r) <= 2 * (m + 3) * U * (aA.T @ np.abs(r)))


@pytest.mark.parametrize("m,n", [(40, 1), (161, 15), (2431, 33), (4865, 97), (3001, 188), (2600, 250)])
def test_lsqr(lsq, handle, m, n):
    g = np.random.default_rng(7 * m + n)
    A = g.standard_normal((m, n))
    b = A @ g.standard_normal(n) + 1e-3 * g.standard_normal(m)
    x = torch.zeros(n, dtype=torch.float64, device="cuda")
    st, _ = lsq.lsq_lsqr(handle, dev(A), dev(b), m, n, min(m, 4 * n), "f64", "f64", "f64", "f64", 1e-13, 1, None, x)
    ref = np.linalg.lstsq(A, b, rcond=None)[0]
    kappa = np.linalg.cond(A)
    assert st == 0
    assert np.linalg.norm(x.cpu().numpy() - ref) <= 20 * kappa * (1e-13 + n * U) * np.linalg.norm(ref)
