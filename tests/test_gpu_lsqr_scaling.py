"""LSQR where squares leave single's range, and the accuracy of its residual norm.

The data are the same up to a power of ten, so the solution is too: to 20 kappa (tol + n u).  The
reported norm is a product of sines from ||b||, each step a few units of rounding: in double
agreement with ||b - A x|| to 1e-10 leaves a factor of 10^3, in single 1e-4 one of 10^2.
"""
import numpy as np
import pytest
import torch

from conftest import dev

pytestmark = pytest.mark.gpu


def lsqr(lsq, handle, A, b, u, tol):
    m, n = A.shape
    x = torch.zeros(n, dtype=torch.float64, device="cuda")
    st, info = lsq.lsq_lsqr(handle, dev(A), dev(b), m, n, min(m, 4 * n), "f64", "f64", u, "f64", tol, 1, None, x)
    assert st == 0 and info.lsqr_flag in (1, 2), (st, info.lsqr_flag)
    return x.cpu().numpy(), info


@pytest.mark.parametrize("sa,sb", [(1.0, 1.0), (1e25, 1e25), (1e-25, 1e-25), (1.0, 1e25), (1.0, 1e-25)])
@pytest.mark.parametrize("m,n", [(2000, 50), (1601, 33), (3001, 188), (1300, 1000)])
def test_double(lsq, handle, m, n, sa, sb):
    g = np.random.default_rng(m + n)
    A = g.standard_normal((m, n))
    b = A @ g.standard_normal(n) + 0.1 * g.standard_normal(m)
    ref = np.linalg.lstsq(A, b, rcond=None)[0]
    kappa = np.linalg.cond(A)
    x, info = lsqr(lsq, handle, A * sa, b * sb, "f64", 1e-13)
    x *= sa / sb
    assert np.linalg.norm(x - ref) <= 20 * kappa * (1e-13 + n * 2.0 ** -53) * np.linalg.norm(ref)
    assert abs(info.lsqr_normr / sb / np.linalg.norm(b - A @ x) - 1) <= 1e-10


@pytest.mark.parametrize("sb", [1.0, 1e22, 1e-28])
@pytest.mark.parametrize("m,n", [(2000, 50), (5001, 33), (3001, 188)])
def test_single(lsq, handle, m, n, sb):
    g = np.random.default_rng(m + n)
    A = g.standard_normal((m, n))
    b = A @ g.standard_normal(n) + 0.1 * g.standard_normal(m)
    ref = np.linalg.lstsq(A, b, rcond=None)[0]
    kappa = np.linalg.cond(A)
    x, info = lsqr(lsq, handle, A, b * sb, "f32", 1e-6)
    x /= sb
    assert np.linalg.norm(x - ref) <= 20 * kappa * (1e-6 + n * 2.0 ** -24) * np.linalg.norm(ref)
    assert abs(info.lsqr_normr / sb / np.linalg.norm(b - A @ x) - 1) <= 1e-4
