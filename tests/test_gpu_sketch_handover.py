"""Sketches whose (tile, split) items do not fill whole waves, so that two CTAs share an item.

One-hot columns make every entry of Y a single product fl_s(G)[i][j], so an accumulator that is lost,
taken twice or loaded into the wrong place shows as a wrong value.  The nonzero rows lie in the first and
last K steps, on both sides of step boundaries and anywhere else.  One to three column groups, one
and three planes, first parts from no step on (fewer steps in an item than SMs).
"""
import numpy as np
import pytest
import torch

pytestmark = pytest.mark.gpu


@pytest.mark.parametrize("fmt,m,n,s,kchunk", [
    ("bf16", 110_000, 40, 2560, 0), ("f16", 60_001, 520, 2560, 0), ("e4m3", 200_003, 30, 2500, 0),
    ("bf16x3", 110_000, 40, 2560, 8192), ("bf16", 70_000, 1024, 2500, 0), ("f16", 300_017, 100, 1100, 0)])
def test_every_entry_is_its_product(lsq, handle, fmt, m, n, s, kchunk):
    r = np.random.default_rng(m)
    edge = np.concatenate([[0, 1, m - 1, m - 2], np.arange(1, 6) * 64 - 1, np.arange(1, 6) * 64])
    rows = np.unique(np.concatenate([edge, r.choice(m, n + 1, replace=False)]))
    rows = r.permutation(rows)[: n + 1] if rows.size > n + 1 and n >= 100 else rows[: n + 1]
    A = torch.zeros(m, n, dtype=torch.float64, device="cuda")
    A[torch.from_numpy(rows[:n]).cuda(), torch.arange(n, device="cuda")] = 1.0
    b = torch.zeros(m, dtype=torch.float64, device="cuda")
    b[int(rows[n])] = -1.0
    Y = torch.full(((n + 1) * s,), float("nan"), dtype=torch.float64, device="cuda")
    lsq.lsq_sketch(handle, A, b, m, n, s, fmt, "f32", "f32", "f64", 1e-6, 5, {"sketch_kchunk": kchunk} if kchunk else None, Y)
    got = Y.view(n + 1, s)
    gfmt = "bf16" if fmt == "bf16x3" else fmt
    for c in range(n + 1):
        g = torch.empty(s * 4, dtype=torch.float64, device="cuda")
        lsq.lsq_omega(handle, s, int(rows[c]) // 4 * 4, 4, gfmt, 5, g)
        ref = g.view(s, 4)[:, int(rows[c]) % 4] * (1.0 if c < n else -1.0) / np.sqrt(s)
        assert torch.all((got[c] - ref).abs() <= 4 * 2.0 ** -53 * ref.abs()), (c, int(rows[c]))
