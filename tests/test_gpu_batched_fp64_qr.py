"""The grouped batch with u_p = double: a problem's bits do not depend on the rest of the batch, whichever of
the others has the largest sketch (s at most 512, and past it).
"""
import pytest
import torch

from conftest import dev
from lsq_synth import randsvd_problem

pytestmark = pytest.mark.gpu

SHAPES = [(3000, 32, 128), (4100, 128, 512), (2500, 77, 511), (7000, 150, 513), (5000, 250, 1000)]   # m, n, s


def solve(lsq, handle, data, sel):
    out = []
    for k in sel:
        m, n, s = SHAPES[k]
        A, b = data[k]
        x, r = (torch.zeros(v, dtype=torch.float64, device="cuda") for v in (n, m))
        out.append(dict(A=A, b=b, m=m, n=n, s=s, seed=k, x=x, r=r))
    st, sts, _ = lsq.lsq_lsir_batched(handle, out, "bf16x3", "f64", "f32", "f64", 1e-6)
    assert st == 0 and all(v == 0 for v in sts), sts
    return out


def test_result_does_not_depend_on_the_largest_sketch(lsq, handle):
    data = []
    for k, (m, n, s) in enumerate(SHAPES):
        P = randsvd_problem(m, n, 1e3, rho=1e-3, seed=300 + k)
        data.append((dev(P.A), dev(P.b)))
    alone = [solve(lsq, handle, data, [k])[0] for k in range(len(SHAPES))]
    for sel in ([0, 1, 2], [0, 3], [1, 4, 2], [4, 3, 2, 1, 0]):
        for k, p in zip(sel, solve(lsq, handle, data, sel)):
            assert torch.equal(p["x"], alone[k]["x"]) and torch.equal(p["r"], alone[k]["r"]), (sel, k)
