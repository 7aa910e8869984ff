"""LSQR solves of one iteration at large n substitute with R instead of forming R^-1: by the cap on the
iterations, or since the start satisfies the tolerance.  From the exact factor one iteration gives the
solution, to 20 (tol + n u); a start within the tolerance stays within kappa tol.
"""
import numpy as np
import pytest
import torch

from conftest import colmajor, dev

pytestmark = pytest.mark.gpu
TOL, U = 1e-6, 2.0 ** -24


def problem(n):
    m = n + n // 2
    g = np.random.default_rng(n)
    A = g.standard_normal((m, n)) / np.sqrt(m) + 2 * np.eye(m, n)
    R = np.linalg.qr(A, mode="r")
    return A, g.standard_normal(n), R * np.where(np.diag(R) < 0, -1.0, 1.0)[:, None]


def solve(lsq, handle, A, b, R, opts):
    m, n = A.shape
    x = torch.zeros(n, dtype=torch.float64, device="cuda")
    _, info = lsq.lsq_lsqr(handle, dev(A), dev(b), m, n, n, "f32", "f32", "f32", "f64", TOL, 1,
                           dict(opts, R_in=dev(colmajor(R)), no_graph=1), x)
    return x.cpu().numpy(), info


@pytest.mark.parametrize("n", [639, 640, 641, 704, 1000, 1023, 1024])
def test_one_iteration(lsq, handle, n):
    A, xt, R = problem(n)
    b = A @ xt + 1e-3 * np.random.default_rng(1).standard_normal(A.shape[0])
    ref = np.linalg.lstsq(A, b, rcond=None)[0]
    launches = {}
    for cap in (1, 2):
        x, info = solve(lsq, handle, A, b, R, {"lsqr_maxit": cap})
        assert np.linalg.norm(x - ref) <= 20 * (TOL + n * U) * np.linalg.norm(ref), cap
        launches[cap] = info.gpu_launches
    # substituting: one launch a step instead of two (a batch of eight and the first), and no inverse
    assert launches[2] - launches[1] == (0 if n < 640 else 8 + 1 + 1), launches


@pytest.mark.parametrize("n", [639, 640, 1000])
def test_start_within_the_tolerance(lsq, handle, n):
    A, xt, R = problem(n)
    kappa = np.linalg.cond(A)
    start = xt * (1 + 1e-8)
    few, info = solve(lsq, handle, A, A @ xt, R, {"x0_in": dev(start)})
    assert info.lsqr_its == 1 and info.lsqr_flag == 1
    assert np.linalg.norm(few - xt) <= 20 * kappa * (TOL + n * U) * np.linalg.norm(xt)
    far, more = solve(lsq, handle, A, A @ xt, R, {})
    assert np.linalg.norm(far - xt) <= 20 * kappa * (TOL + n * U) * np.linalg.norm(xt)
    per_step = 8 * 4 if n < 640 else 8 * 3   # launches of a batch: pass, column sums, the step
    assert info.gpu_launches - more.gpu_launches == (per_step + (0 if n < 640 else -2)
                                                     - 8 * 4 * (-(-more.lsqr_its // 8))), (info.gpu_launches, more.gpu_launches)
