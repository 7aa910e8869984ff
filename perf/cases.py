"""What is timed: calls of the public entry points over the sizes, precisions and options this solver is used with.

A case names the entry point (``kind``), the sizes m, n, s, the precisions (u_s sketch, u_p QR, u_w working, u_r
residual) and the conditioning of its problem.  Problems are drawn like the paper's randsvd matrices: A = U diag(sigma)
V^T with sigma geometric from 1 to 1/kappa and V Haar; U is a Gaussian m x n matrix over sqrt(m), which has nearly
orthonormal columns for m >> n and is quick to draw.  Entries of A have full FP64 significands.  b = A x_true + noise
of relative size rho.

The calls write FP64 buffers whatever the precision they were computed in.  Where that was single (u_w or u_p single; a
tensor-core sketch, which accumulates in FP32) the program keeps the result in single, as the method delivers it
(forward errors of a few units in the last place of single); FP64 factors and solves in double stay FP64.
"""
import math
import random

import torch

import paper_2410_06319_gb300 as lsq

F32, F64 = torch.float32, torch.float64


def listed():
    return [
        # the paper's experiment (Sec. 5): one small problem, where launches and host round trips are the time
        dict(name="lsir_m1000_n100", kind="lsir", m=1000, n=100, s=400, u_s="bf16", u_p="f32", u_w="f32", u_r="f64",
             kappa=1e2, rho=1e-1, tol=1e-6),
        # the plain method, everything in FP64: sketch, QR and LSQR to 1e-14 on a small problem
        dict(name="lsqr_f64_m2000_n50", kind="lsqr", m=2000, n=50, s=200, u_s="f64", u_p="f64", u_w="f64", u_r="f64",
             kappa=1e3, rho=1e-4, tol=1e-14),
        # u = double with double-double residuals (Table 4's setting) at odd sizes
        dict(name="lsir_f64x2_m20011_n187", kind="lsir", m=20011, n=187, s=748, u_s="bf16x3", u_p="f64", u_w="f64",
             u_r="f64x2", kappa=1e4, rho=1e-3, tol=1e-12),
        # the middle configuration, whole: sketch, QR, LSQR and refinement
        dict(name="lsir_m100000_n500", kind="lsir", m=100_000, n=500, s=2000, u_s="bf16x3", u_p="f32", u_w="f32",
             u_r="f64", kappa=1e6, rho=1e-3, tol=1e-6),
        # many uneven problems in one call
        dict(name="batched_32", kind="batched", count=32, m_lo=5000, m_hi=200_000, n_lo=32, n_hi=256, sizes=4,
             u_s="bf16", u_p="f32", u_w="f32", u_r="f64", kappa=50.0, rho=1e-3, tol=1e-6),
        # the LSQR solve alone (sketch, QR, LSQR) at the kappa = 10 configuration, a size off every tile
        dict(name="lsqr_m600011_n601", kind="lsqr", m=600_011, n=601, s=1803, u_s="e4m3", u_p="f32", u_w="f32",
             u_r="f64", kappa=10.0, rho=1e-2, tol=1e-6),
        # one refinement step (residual, two solves per FGMRES iteration, Arnoldi, update) on a long problem
        dict(name="ir_step_m1000000_n1000", kind="ir_step", m=1_000_000, n=1000, s=4000, u_s="bf16x3", u_p="f64",
             u_w="f32", u_r="f64", kappa=1e4, rho=1e-3, tol=1e-6),
        # the sketch alone: single-term BF16 at the middle size, FP16 and the three-term BF16 split at the large one
        dict(name="sketch_bf16_m100000_n500", kind="sketch", m=100_000, n=500, s=2000, u_s="bf16", kappa=1e2, rho=1e-3),
        dict(name="sketch_f16_m1000000_n1000", kind="sketch", m=1_000_000, n=1000, s=3000, u_s="f16", kappa=1e3,
             rho=1e-2),
        dict(name="sketch_bf16x3_m1000000_n1000", kind="sketch", m=1_000_000, n=1000, s=4000, u_s="bf16x3", kappa=1e5,
             rho=1e-3),
        # the QR of a sketch in both precisions (one sketch is factored again in another precision or for another b)
        dict(name="qr_f32_s2000_n500", kind="qr", n=500, s=2000, u_p="f32", kappa=10.0),
        dict(name="qr_f64_s4000_n1000", kind="qr", n=1000, s=4000, u_p="f64", kappa=1e4),
    ]


def _log(rng, lo, hi):
    return math.exp(rng.uniform(math.log(lo), math.log(hi)))


def draw(rng):
    kind = rng.choice(["lsir", "lsir", "lsqr", "ir_step", "sketch", "sketch", "qr", "batched"])
    if kind == "batched":
        return dict(kind=kind, count=rng.randint(2, 32), m_lo=rng.randint(600, 5000), m_hi=rng.randint(20_000, 200_000),
                    n_lo=rng.randint(16, 40), n_hi=rng.randint(64, 256), sizes=rng.randint(0, 10**6),
                    u_s=rng.choice(["bf16", "f16", "bf16x3"]), u_p="f32", u_w="f32", u_r="f64",
                    kappa=_log(rng, 5.0, 50.0), rho=_log(rng, 1e-4, 1e-1), tol=1e-6)
    n = int(_log(rng, 24, 1000))
    if kind == "qr":
        # x_s is asked for beside R: its error is about kappa times the unit roundoff of the factorization
        u_p = rng.choice(["f32", "f64"])
        return dict(kind=kind, n=n, s=rng.randint(2 * n, 4 * n), u_p=u_p, kappa=_log(rng, 4, 20 if u_p == "f32" else 1e4))
    m = int(_log(rng, 10 * n, 10**6))
    s = min(rng.choice([2, 3, 4]) * n + rng.choice([0, 0, rng.randint(1, n)]), m, 4000)
    if kind == "sketch":
        return dict(kind=kind, m=m, n=n, s=s, u_s=rng.choice(["bf16", "f16", "e4m3", "bf16x3"]), kappa=_log(rng, 10, 1e5),
                    rho=_log(rng, 1e-4, 1e-1))
    if kind != "ir_step" and rng.random() < 0.25:   # u = double; its FP64 products are meant for moderate sizes
        m = int(_log(rng, 10 * min(n, 200), 30_000))
        n = min(n, 200, m // 10)
        u = dict(u_s="bf16x3", u_p="f64", u_w="f64", u_r=rng.choice(["f64", "f64x2"]), tol=1e-12)
        return dict(kind=kind, m=m, n=n, s=4 * n, kappa=_log(rng, 10, 1e4), rho=_log(rng, 1e-4, 1e-1), **u)
    u = dict(u_s="bf16x3", u_p=rng.choice(["f32", "f64"]), u_w="f32", u_r="f64", tol=1e-6)
    # LSQR alone in single is for well-conditioned problems: its error is about kappa times the unit roundoff
    kappa = _log(rng, 4, 20) if kind == "lsqr" else _log(rng, 10, 1e5)
    return dict(kind=kind, m=m, n=n, s=max(s, min(3 * n, m)), kappa=kappa, rho=_log(rng, 1e-4, 1e-1), **u)


# ------------------------------------------------------------------------------------------------- inputs
_handle = []


def _lsq_handle():
    """The program's one handle (its workspace serves every call, as in a program that solves many problems)."""
    if not _handle:
        _handle.append(lsq.Handle())
    return _handle[0]


def _factor(n, kappa, g):
    """diag(sigma) V^T in FP64."""
    v, r = torch.linalg.qr(torch.randn(n, n, generator=g, device="cuda", dtype=F64))
    v = v * torch.where(torch.diagonal(r) < 0, -1.0, 1.0)
    sigma = float(kappa) ** (-torch.arange(n, device="cuda", dtype=F64) / max(1, n - 1))
    return sigma[:, None] * v.T


def _rows(m, w, g):
    """m rows of a Gaussian matrix over sqrt(m) times w, with full FP64 significands."""
    n = w.shape[0]
    a = torch.empty(m, n, device="cuda", dtype=F64)
    w32 = (w / math.sqrt(m)).to(F32)
    for i in range(0, m, 1 << 17):
        k = min(m - i, 1 << 17)
        c = torch.randn(k, n, generator=g, device="cuda") @ w32
        low = torch.rand(k, n, generator=g, device="cuda").sub_(0.5).mul_(2.0 ** -24).mul_(c)
        a[i:i + k] = c.double() + low.double()
    return a


def _problem(m, n, kappa, rho, g):
    a = _rows(m, _factor(n, kappa, g), g)
    x = torch.randn(n, generator=g, device="cuda", dtype=F64)
    ax = a @ x
    e = torch.randn(m, generator=g, device="cuda", dtype=F64)
    e *= rho / math.sqrt(1 - rho * rho) * torch.linalg.norm(ax) / torch.linalg.norm(e)
    return a, ax + e, x


def _gen(seed):
    g = torch.Generator(device="cuda")
    g.manual_seed(int(seed))
    return g


def _sizes(case):
    """(m, n) of each problem of a batch."""
    r = random.Random(case["sizes"])
    for _ in range(case["count"]):
        n = r.randint(case["n_lo"], case["n_hi"])
        yield max(10 * n, r.randint(case["m_lo"], case["m_hi"])), n


def prepare(case, seed):
    g = _gen(seed)
    st = dict(case=case, seed=int(seed), h=_lsq_handle())
    zeros = lambda *k: torch.zeros(*k, device="cuda", dtype=F64)  # noqa: E731
    if case["kind"] == "batched":
        st["probs"] = []
        for k, (m, n) in enumerate(_sizes(case)):
            a, b, _ = _problem(m, n, case["kappa"], case["rho"], g)
            st["probs"].append(dict(A=a, b=b, m=m, n=n, s=4 * n, seed=seed + k, x=zeros(n), r=zeros(m)))
        return st
    n = case["n"]
    if case["kind"] == "qr":   # a sketch as lsq_sketch leaves it: s x (n + 1), column-major
        a, b, _ = _problem(case["s"], n, case["kappa"], 0.1, g)
        st.update(Y=torch.cat([a, b[:, None]], 1).T.contiguous(), R=zeros(n, n), xs=zeros(n))
        return st
    m = case["m"]
    st["A"], st["b"], x = _problem(m, n, case["kappa"], case["rho"], g)
    if case["kind"] == "sketch":
        st["Y"] = zeros(n + 1, case["s"])
    elif case["kind"] == "ir_step":
        # R of a sketch: the rows of A are alike, so 4n of them have the law of a Gaussian sketch; x and r are what an
        # LSQR start in single leaves
        k = min(m, 4 * n)
        r = torch.linalg.qr(st["A"][:k] * math.sqrt(m / k), mode="r").R
        st["R"] = (r * torch.where(torch.diagonal(r) < 0, -1.0, 1.0)[:, None]).T.contiguous()
        st["x0"] = x * (1 + 1e-4 * torch.randn(n, generator=g, device="cuda", dtype=F64))
        st["r0"] = (st["b"] - st["A"] @ st["x0"]).float().double()
        st.update(x=zeros(n), r=zeros(m))
    else:
        st.update(x=zeros(n), r=zeros(m))
    return st


# --------------------------------------------------------------------------------------------------- calls
def run(st):
    c, h = st["case"], st["h"]
    if c["kind"] == "batched":
        lsq.lsq_lsir_batched(h, st["probs"], c["u_s"], c["u_p"], c["u_w"], c["u_r"], c["tol"])
        return [dict(x=p["x"].float(), r=p["r"].float()) for p in st["probs"]]
    if c["kind"] == "qr":
        lsq.lsq_qr_r(h, None, None, max(c["s"], c["n"]), c["n"], c["s"], "f64", c["u_p"], "f64", "f64", 1.0, 0,
                     dict(Y_in=st["Y"]), st["R"], st["xs"])
        out = F32 if c["u_p"] == "f32" else F64
        return dict(R=st["R"].to(out), xs=st["xs"].to(out))
    m, n, s = c["m"], c["n"], c["s"]
    if c["kind"] == "sketch":
        lsq.lsq_sketch(h, st["A"], st["b"], m, n, s, c["u_s"], "f32", "f32", "f64", 1.0, st["seed"], None, st["Y"])
        return st["Y"].float()
    args = (h, st["A"], st["b"], m, n, s, c["u_s"], c["u_p"], c["u_w"], c["u_r"], c["tol"], st["seed"], None)
    out = F32 if c["u_w"] == "f32" else F64
    if c["kind"] == "lsqr":
        lsq.lsq_lsqr(*args, st["x"])
        return st["x"].to(out)
    if c["kind"] == "ir_step":
        st["x"].copy_(st["x0"])
        st["r"].copy_(st["r0"])
        lsq.lsq_ir_step(*args, st["R"], st["x"], st["r"])
    else:
        lsq.lsq_lsir(*args, st["x"], st["r"])
    return dict(x=st["x"].to(out), r=st["r"].to(out))


#: iterations that a good sketch leaves to do (kappa(A R^-1) about 3 at s = 4n; Tables 1 to 4 of the paper)
LSQR_ITS = {"f32": 16, "f64": 32}
FGMRES_ITS = {"f32": 40, "f64": 60}


def _work(c, m, n, s):
    sketch = 2.0 * s * m * (n + 1) * (3 if c["u_s"] == "bf16x3" else 1)
    qr = 2.0 * n * n * (s - n / 3)
    its = {"lsqr": LSQR_ITS[c["u_w"]], "ir_step": FGMRES_ITS[c["u_w"]] / 2,
           "lsir": LSQR_ITS[c["u_w"]] + FGMRES_ITS[c["u_w"]]}[c["kind"] if c["kind"] != "batched" else "lsir"]
    flops = its * 4.0 * m * n + (0 if c["kind"] == "ir_step" else sketch + qr)
    return 8.0 * m * n + 8.0 * m + 8.0 * n + (8.0 * m if c["kind"] != "lsqr" else 0), flops


def work(case):
    c = case
    if c["kind"] == "batched":
        w = [_work(c, m, n, 4 * n) for m, n in _sizes(c)]
        return dict(bytes=sum(x[0] for x in w), flops=sum(x[1] for x in w))
    n = c["n"]
    if c["kind"] == "qr":
        return dict(bytes=8.0 * c["s"] * (n + 1) + 8.0 * n * n, flops=2.0 * n * n * (c["s"] - n / 3))
    m, s = c["m"], c["s"]
    if c["kind"] == "sketch":
        return dict(bytes=8.0 * m * (n + 1) + 8.0 * s * (n + 1),
                    flops=2.0 * s * m * (n + 1) * (3 if c["u_s"] == "bf16x3" else 1))
    b, f = _work(c, m, n, s)
    return dict(bytes=b, flops=f)


# ------------------------------------------------------------------------------------------ 64-bit results
def _least_squares(a, b):
    """The solution by the normal equations, refined in FP64 (kappa^2 u < 1 here)."""
    d = torch.linalg.norm(a, dim=0)
    l = torch.linalg.cholesky((a.T @ a) / d[:, None] / d[None, :])
    x = torch.zeros(a.shape[1], device="cuda", dtype=F64)
    for _ in range(6):
        x = x + torch.cholesky_solve(((a.T @ (b - a @ x)) / d)[:, None], l)[:, 0] / d
    return x, b - a @ x


def _philox(c0, c1, k0, k1):
    """Philox4x32-10 of the counters (c0, c1, 0, 0); 32-bit words in int64 (c0 < 2^32)."""
    m32 = 0xFFFFFFFF
    c = [c0, c1, torch.zeros_like(c0), torch.zeros_like(c0)]
    for _ in range(10):
        p0, p1 = 0xD2511F53 * c[0], 0xCD9E8D57 * c[2]
        c = [((p1 >> 32) & m32) ^ c[1] ^ k0, p1 & m32, ((p0 >> 32) & m32) ^ c[3] ^ k1, p0 & m32]
        k0, k1 = (k0 + 0x9E3779B9) & m32, (k1 + 0xBB67AE85) & m32
    return c


def _gauss(s, j0, cols, seed, dev="cuda"):
    """G[:s, j0:j0 + cols] (cols and j0 multiples of 4): Box-Muller of the Philox words (a, b), U1 = (a + 1) / 2^32."""
    q = torch.arange(j0 // 4, (j0 + cols) // 4, device=dev)[None, :].expand(s, -1).contiguous()
    i = torch.arange(s, device=dev)[:, None].expand_as(q).contiguous()
    w = _philox(q, i, seed & 0xFFFFFFFF, (seed >> 32) & 0xFFFFFFFF)
    g = []
    for a, b in ((w[0], w[1]), (w[2], w[3])):
        rad = torch.sqrt(-2.0 * torch.log((a + 1).double() * 2.0 ** -32))
        ang = b.double() * (2.0 ** -32 * 2 * math.pi)
        g += [rad * torch.cos(ang), rad * torch.sin(ang)]
    return torch.stack(g, -1).reshape(s, cols)


def _sketch(a, b, s, u_s, seed):
    """s^-1/2 fl_s(G) [A | b] in FP64: the sketch matrix as it is defined, the data as given."""
    m, n = a.shape
    to = {"bf16": torch.bfloat16, "bf16x3": torch.bfloat16, "f16": torch.float16, "e4m3": torch.float8_e4m3fn,
          "f64": F64}[u_s]
    y = torch.zeros(s, n + 1, device="cuda", dtype=F64)
    for j in range(0, m, 8192):
        k = min(8192, m - j)
        g = _gauss(s, j, (k + 3) // 4 * 4, seed)[:, :k]
        g = g.to(to).double() if to != F64 else g
        y[:, :n].addmm_(g, a[j:j + k])
        y[:, n].addmv_(g, b[j:j + k])
    return y.T.contiguous() / math.sqrt(s)


def exact(case, seed):
    c = case
    st = prepare(case, seed)
    if c["kind"] == "batched":
        return [dict(zip("xr", _least_squares(p["A"], p["b"]))) for p in st["probs"]]
    if c["kind"] == "qr":
        y = st["Y"].T
        q, r = torch.linalg.qr(y[:, :c["n"]])
        sg = torch.where(torch.diagonal(r) < 0, -1.0, 1.0)
        r, z = r * sg[:, None], (q.T @ y[:, c["n"]]) * sg
        return dict(R=r.T.contiguous(), xs=torch.linalg.solve_triangular(r, z[:, None], upper=True)[:, 0])
    if c["kind"] == "sketch":
        return _sketch(st["A"], st["b"], c["s"], c["u_s"], st["seed"])
    x, r = _least_squares(st["A"], st["b"])
    return x if c["kind"] == "lsqr" else dict(x=x, r=r)
