"""The Arnoldi step's forms (one cluster, grid with w and the basis in shared memory, modified
Gram-Schmidt in blocks of eight) where their ranges end: lengths m + n about 16 rows a CTA, the cluster's
limit of 2048 rows and the slab's, with one column and with many.  Every form must lead to the
solution within the 4u target, and the forms' iteration counts must agree.
"""
import numpy as np
import pytest
import torch

from conftest import dev
from lsq_synth import randsvd_problem
from oracle import exact

pytestmark = pytest.mark.gpu

U32 = 2.0 ** -24


def zeros(k):
    return torch.zeros(k, dtype=torch.float64, device="cuda")


@pytest.mark.parametrize("length,n", [(3, 1), (17, 3), (64, 5), (65, 5), (1025, 40), (2047, 33), (2048, 33), (2049, 33),
                                      (9729, 60), (20011, 17)])
def test_every_form_reaches_the_solution(lsq, handle, length, n):
    m = length - n
    P = randsvd_problem(m, n, 1e3 if n > 1 else 1.0, rho=1e-2, seed=length)
    xstar, rstar = exact.reference_solution(P.A, P.b)
    its = []
    for form in (0, 1, 2, 3):
        x, r = zeros(n), zeros(m)
        st, info = lsq.lsq_lsir(handle, dev(P.A), dev(P.b), m, n, min(m, 4 * n), "bf16x3", "f32", "f32", "f64", 1e-6, 7,
                                {"arnoldi": form}, x, r)
        ex, er = exact.forward_errors(x.cpu().numpy(), r.cpu().numpy(), xstar, rstar)
        assert st == 0 and info.ir_converged == 1, (form, st)
        assert ex <= 4 * U32 and er <= 4 * U32, (form, ex, er)
        its.append(info.gmres_its_total)
    assert max(its) - min(its) <= 4, its


@pytest.mark.parametrize("u_r", ["f64", "f64x2"])
@pytest.mark.parametrize("length,n", [(2048, 20), (2049, 20), (6007, 101)])
def test_fp64_products(lsq, handle, length, n, u_r):
    m = length - n
    P = randsvd_problem(m, n, 1e2, rho=1e-2, seed=length + 1)
    xstar, rstar = exact.reference_solution(P.A, P.b)
    sols = []
    for form in (1, 2, 3):
        x, r = zeros(n), zeros(m)
        st, info = lsq.lsq_lsir(handle, dev(P.A), dev(P.b), m, n, 4 * n, "bf16x3", "f64", "f64", u_r, 1e-12, 7,
                                {"arnoldi": form}, x, r)
        ex, _ = exact.forward_errors(x.cpu().numpy(), r.cpu().numpy(), xstar, rstar)
        assert ex <= 1e2 * n * 2.0 ** -53 * 10, (form, ex)


@pytest.mark.parametrize("cap", [1, 31, 32, 33, 64, 65, 97, 127])
def test_back_substitution_lengths(lsq, handle, cap):
    """A tolerance that is never reached makes every correction take `cap` columns: the triangular
    system of the update ends at every place of a register and of a warp."""
    m, n = 700, 150
    P = randsvd_problem(m, n, 1e2, rho=1e-2, seed=cap)
    xstar, rstar = exact.reference_solution(P.A, P.b)
    x, r = zeros(n), zeros(m)
    st, info = lsq.lsq_lsir(handle, dev(P.A), dev(P.b), m, n, 600, "bf16x3", "f32", "f32", "f64", 1e-6, 7,
                            {"gmres_maxit": cap, "gmres_tol": 1e-30, "ir_maxit": 6}, x, r)
    assert info.gmres_its[0] == cap
    ex, er = exact.forward_errors(x.cpu().numpy(), r.cpu().numpy(), xstar, rstar)
    if cap > 30:
        assert ex <= 4 * U32 and er <= 4 * U32, (ex, er)
    else:   # one column a correction: each must not increase the error of LSQR's start
        assert np.isfinite(ex) and ex <= 1e-3
