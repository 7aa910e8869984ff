"""The QR of a sketch where its column blocks and row groups end: n mod 8 (FP32) and mod 4 (FP64), a
block that holds only the right-hand side, s at and past the rows a CTA's registers hold.

R^T R = Y^T Y to 8 (n + sqrt(s)) u and R x_s = c to the same times the condition of a Gaussian
matrix with s >= 2n (below 6; nearer to square, the condition itself).
"""
import numpy as np
import pytest
import torch

from conftest import colmajor, dev, from_colmajor

pytestmark = pytest.mark.gpu

F32 = [(2, 1), (3, 1), (33, 7), (64, 8), (65, 9), (511, 16), (512, 127), (513, 128), (1024, 31), (1025, 255), (2048, 401),
       (2049, 15), (2300, 1023), (3999, 512), (4096, 24), (4097, 33)]
F64 = [(2, 1), (9, 3), (16, 4), (33, 5), (511, 61), (512, 64), (513, 63), (255, 64), (257, 128), (1024, 251), (1025, 12),
       (1030, 1024), (2047, 700), (2048, 3), (2049, 130), (4095, 260), (4096, 2), (4097, 9)]


@pytest.mark.parametrize("up,s,n", [("f32",) + c for c in F32] + [("f64",) + c for c in F64])
def test_factor_and_solution(lsq, handle, up, s, n):
    Y = np.random.default_rng(s + n).standard_normal((s, n + 1))
    Y[:, : n // 2] *= 1e3
    R = torch.zeros(n * n, dtype=torch.float64, device="cuda")
    xs = torch.zeros(n, dtype=torch.float64, device="cuda")
    lsq.lsq_qr_r(handle, None, None, max(s, n), n, s, "f64", up, "f64", "f64", 1.0, 0, {"Y_in": dev(colmajor(Y))}, R, xs)
    Rg = from_colmajor(R, n, n)
    tol = 8 * (n + np.sqrt(s)) * (2.0 ** -24 if up == "f32" else 2.0 ** -53)
    assert np.all(np.tril(Rg, -1) == 0) and np.all(np.diag(Rg) >= 0)
    d = np.linalg.norm(Y[:, :n], axis=0)      # columns scaled apart: the error is column by column
    G = (Y[:, :n] / d).T @ (Y[:, :n] / d)
    assert np.linalg.norm((Rg / d).T @ (Rg / d) - G) <= tol * np.linalg.norm(G)
    ref = np.linalg.lstsq(Y[:, :n] / d, Y[:, n], rcond=None)[0]
    got = xs.cpu().numpy() * d
    kappa = 6.0 if s >= 2 * n else np.linalg.cond(Y[:, :n] / d)
    assert np.linalg.norm(got - ref) <= kappa ** 2 * tol * (np.linalg.norm(ref) + np.linalg.norm(Y[:, n]))


@pytest.mark.parametrize("up", ["f32", "f64"])
def test_zero_columns_stay_zero(lsq, handle, up):
    s, n = 200, 21
    Y = np.random.default_rng(1).standard_normal((s, n + 1))
    Y[:, [0, 8, 20]] = 0.0
    R = torch.zeros(n * n, dtype=torch.float64, device="cuda")
    xs = torch.zeros(n, dtype=torch.float64, device="cuda")
    try:
        lsq.lsq_qr_r(handle, None, None, s, n, s, "f64", up, "f64", "f64", 1.0, 0, {"Y_in": dev(colmajor(Y))}, R, xs)
    except lsq.LsqError:
        pass   # a singular R is reported; the factor is written all the same
    Rg = from_colmajor(R, n, n)
    u = 2.0 ** -24 if up == "f32" else 2.0 ** -53
    assert np.linalg.norm(Rg.T @ Rg - Y[:, :n].T @ Y[:, :n]) <= 8 * (n + np.sqrt(s)) * u * np.linalg.norm(Y[:, :n]) ** 2
    assert np.all(Rg[:, [0, 8, 20]] == 0)
