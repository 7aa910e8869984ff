"""The batch's row pass where its ring and its pieces end: rows of 1 to 64 float4, fewer rows than warps,
one row pair more or less than the ring holds, one row past an item.  Each problem must reach the 4u
target of the single solve.
"""
import pytest
import torch

from conftest import dev
from lsq_synth import randsvd_problem
from oracle import exact

pytestmark = pytest.mark.gpu

U32 = 2.0 ** -24


def zeros(k):
    return torch.zeros(k, dtype=torch.float64, device="cuda")


@pytest.mark.parametrize("shapes", [
    [(5, 1), (8, 2), (9, 3), (16, 4), (17, 5), (31, 6), (33, 7), (49, 8)],
    [(1023, 31), (1024, 32), (1025, 33), (1040, 127), (1041, 128), (1057, 129)],
    [(2047, 255), (2049, 256), (3073, 12), (1100, 250)]])
def test_every_problem_reaches_the_solution(lsq, handle, shapes):
    Ps, probs = [], []
    for k, (m, n) in enumerate(shapes):
        P = randsvd_problem(m, n, 10.0 if n > 1 else 1.0, rho=1e-2, seed=31 * m + n)
        Ps.append(P)
        probs.append(dict(A=dev(P.A), b=dev(P.b), m=m, n=n, s=min(m, 4 * n), seed=k, x=zeros(n), r=zeros(m)))
    st, sts, infos = lsq.lsq_lsir_batched(handle, probs, "bf16x3", "f32", "f32", "f64", 1e-6)
    assert st == 0 and all(v == 0 for v in sts), sts
    for P, pr, inf in zip(Ps, probs, infos):
        xstar, rstar = exact.reference_solution(P.A, P.b)
        ex, er = exact.forward_errors(pr["x"].cpu().numpy(), pr["r"].cpu().numpy(), xstar, rstar)
        assert inf.ir_converged == 1 and ex <= 4 * U32 and er <= 4 * U32, (P.meta, ex, er)
