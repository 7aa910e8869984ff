"""The products with R^-1 inside LSQR and FGMRES, at the sizes where rows, warps and 16-byte pieces end.

LSQR from the exact triangular factor takes one or two steps, so its result shows an entry of R^-1
that is missing or misplaced at once; LSIR must reach the 4u target with every size.  Tolerances:
LSQR stops at tol; its result is within kappa (tol + n u) of the solution.
"""
import numpy as np
import pytest
import torch

from conftest import colmajor, dev
from lsq_synth import randsvd_problem
from oracle import exact

pytestmark = pytest.mark.gpu


def zeros(k):
    return torch.zeros(k, dtype=torch.float64, device="cuda")


@pytest.mark.parametrize("u", ["f32", "f64"])
@pytest.mark.parametrize("n", [1, 2, 7, 8, 9, 31, 32, 33, 64, 65, 255, 257])
def test_lsqr_with_the_exact_factor(lsq, handle, u, n):
    m = 4 * n + 37
    P = randsvd_problem(m, n, 10.0 if n > 1 else 1.0, rho=1e-3, seed=n)
    R = np.linalg.qr(P.A, mode="r")
    R = R * np.where(np.diag(R) < 0, -1.0, 1.0)[:, None]
    tol, ur = (1e-6, 2.0 ** -24) if u == "f32" else (1e-13, 2.0 ** -53)
    x = zeros(n)
    st, info = lsq.lsq_lsqr(handle, dev(P.A), dev(P.b), m, n, 2 * n, "f32", u, u, "f64", tol, 1,
                            {"R_in": dev(colmajor(R))}, x)
    xstar, _ = exact.reference_solution(P.A, P.b)
    assert st == 0 and info.lsqr_its <= 4
    assert np.linalg.norm(x.cpu().numpy() - xstar) <= 20 * (tol + n * ur) * np.linalg.norm(xstar)


@pytest.mark.parametrize("m,n", [(1100, 1024), (1500, 1000)])
def test_lsqr_with_the_exact_factor_at_the_largest_sizes(lsq, handle, m, n):
    g = np.random.default_rng(n)
    A = g.standard_normal((m, n)) / np.sqrt(m) + np.eye(m, n)
    xt = g.standard_normal(n)
    b = A @ xt
    R = np.linalg.qr(A, mode="r")
    R = R * np.where(np.diag(R) < 0, -1.0, 1.0)[:, None]
    kappa = np.linalg.cond(R)
    x = zeros(n)
    st, info = lsq.lsq_lsqr(handle, dev(A), dev(b), m, n, n, "f32", "f32", "f32", "f64", 1e-6, 1,
                            {"R_in": dev(colmajor(R))}, x)
    assert st == 0 and info.lsqr_its <= 4
    assert np.linalg.norm(x.cpu().numpy() - xt) <= kappa * 2 * (1e-6 + n * 2.0 ** -24) * np.linalg.norm(xt)


@pytest.mark.parametrize("n", [1, 5, 32, 33, 100])
def test_one_correction_and_the_iterated_refinement_agree(lsq, handle, n):
    """One correction substitutes, several use products: both lead to the solution."""
    m = 20 * n + 11
    P = randsvd_problem(m, n, 100.0 if n > 1 else 1.0, rho=1e-2, seed=50 + n)
    xstar, rstar = exact.reference_solution(P.A, P.b)
    R = np.linalg.qr(P.A, mode="r")
    R = R * np.where(np.diag(R) < 0, -1.0, 1.0)[:, None]
    args = (handle, dev(P.A), dev(P.b), m, n, 4 * n, "bf16x3", "f32", "f32", "f64", 1e-6, 3)
    x, r = zeros(n), zeros(m)
    st, _ = lsq.lsq_lsir(*args, None, x, r)
    ex, er = exact.forward_errors(x.cpu().numpy(), r.cpu().numpy(), xstar, rstar)
    assert st == 0 and ex <= 4 * 2.0 ** -24 and er <= 4 * 2.0 ** -24
    x1 = dev(xstar * (1 + 1e-3))
    r1 = dev(P.b - P.A @ (xstar * (1 + 1e-3)))
    Rd = dev(colmajor(R))
    for _ in range(3):
        lsq.lsq_ir_step(*args, None, Rd, x1, r1)
    ex, er = exact.forward_errors(x1.cpu().numpy(), r1.cpu().numpy(), xstar, rstar)
    assert ex <= 4 * 2.0 ** -24 and er <= 4 * 2.0 ** -24
