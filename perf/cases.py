"""The work a user of the tracker has it do, as measured cases.

Every case is one call (or the few calls a program makes together) through the
public Python entry points of ``paper_2107_01104_gb300``.  Fields are random
divergence-free Fourier fields with a Kolmogorov-like spectrum and unit rms,
tracers are uniform in the box (some sets have left it: positions are
unwrapped).  The sizes are those of the repository's benchmark, tests and
configurations, scaled so that a pass takes from tens of microseconds to tens
of milliseconds.

``kind`` says what a case does:

* ``step``     X_0 -> X_T: ``advance`` by RK2 or Adams-Bashforth steps;
* ``small``    ``interpolate`` and one step of a small set (latency);
* ``coupled``  ``set_field`` and one step: a solver that hands over a new field;
* ``interp``   ``interpolate``: every component, or the gradient (``deriv``);
* ``batched``  ``advance_batched``: several sets of uneven size and kernels;
* ``adjoint``  ``advect`` and its backward pass (autograd);
* ``bin``      ``bin``: the stable block binning.
"""
from __future__ import annotations

import math
from fractions import Fraction

import numpy as np
import torch

import paper_2107_01104_gb300 as trk
from paper_2107_01104_gb300.autograd import advect

TWO_PI = 2.0 * math.pi
FAMILY = {"lagrange": trk.TRK_LAGRANGE, "spline": trk.TRK_SPLINE}
STORAGE = {"f64": trk.TRK_F64, "f32": trk.TRK_F32, "bf16x2": trk.TRK_BF16X2}
SCHEME = {"rk2": trk.TRK_RK2, "ab2": trk.TRK_AB2, "ab3": trk.TRK_AB3, "ab4": trk.TRK_AB4}
ESZ = {"f64": 8, "f32": 4, "bf16x2": 4}


def listed():
    return [
        # the plain method at its smallest: u at the tracers and one RK2 step of 10^4 tracers on 32^3 in
        # float64 (latency and launches)
        dict(name="small_f64", kind="small", N=32, family="lagrange", I=4, m=0, storage="f64", np=10000,
             scheme="rk2", dt=1e-3, steps=1),
        # the headline workload: 2^20 tracers on 256^3 float32, spline I = 6, RK2, re-binned every step
        dict(name="rk2_f32_256", kind="step", N=256, family="spline", I=6, m=2, storage="f32", np=1 << 20,
             scheme="rk2", dt=5e-3, steps=20),
        # the same method in float64 storage and arithmetic (the paper's plain form), an odd count
        dict(name="rk2_f64_128", kind="step", N=128, family="spline", I=6, m=2, storage="f64", np=200003,
             scheme="rk2", dt=5e-3, steps=4),
        # the paper's multi-step scheme on a densely seeded box, short stencil, a restarted run with full history
        dict(name="ab4_dense_128", kind="step", N=128, family="spline", I=4, m=1, storage="f32", np=777777,
             scheme="ab4", dt=4e-3, steps=8),
        # the paper's production density (1.5e-3 tracers per cell)
        dict(name="rk2_sparse_512", kind="step", N=512, family="spline", I=6, m=2, storage="f32", np=200000,
             scheme="rk2", dt=2.5e-3, steps=10),
        # one particle step per step of the flow solver: a new field every call
        dict(name="coupled_ab2_256", kind="coupled", N=256, family="spline", I=6, m=2, storage="f32", np=300001,
             scheme="ab2", dt=2.5e-3, steps=1),
        # u of a large set with the widest kernel, 1/8 tracer per cell
        dict(name="interp_u_f32_512", kind="interp", N=512, family="spline", I=8, m=3, storage="f32", np=1 << 24,
             C=3, deriv=False, out="f32"),
        # u and its spectral gradient (12 components) from split-bf16 storage
        dict(name="interp_12c_bf16_256", kind="interp", N=256, family="spline", I=8, m=3, storage="bf16x2",
             np=1 << 21, C=12, deriv=False, out="f32"),
        # the velocity gradient by kernel derivatives, an odd count
        dict(name="interp_grad_f32_256", kind="interp", N=256, family="lagrange", I=6, m=0, storage="f32",
             np=999983, C=3, deriv=True, out="f32"),
        # eight sets of uneven size, kernels cycling I = 4, 6, 8, outputs of 3 or 9 components
        dict(name="batched_256", kind="batched", N=256, storage="f32", nsets=8, smallest=1000, largest=2000000,
             dt=2.5e-3, steps=6),
        # gradient of a loss through RK2 steps with respect to the tracers (float32 parameters, as an
        # optimiser keeps them) and the field
        dict(name="adjoint_256", kind="adjoint", N=256, family="spline", I=6, m=2, storage="f32", np=1 << 22,
             dt=5e-3, steps=5),
        # the stable block binning on its own
        dict(name="bin_256", kind="bin", N=256, np=(1 << 22) + 3),
    ]


# --------------------------------------------------------------------------
# Drawn cases
# --------------------------------------------------------------------------
def _log_int(rng, lo, hi):
    return int(round(math.exp(rng.uniform(math.log(lo), math.log(hi)))))


def _draw_once(rng):
    kind = rng.choice(["small", "step", "step", "step", "coupled", "interp", "interp", "batched", "adjoint", "bin"])
    N = rng.choice([16, 32, 64] if kind == "small" else [32, 64, 128, 256, 512])
    I = rng.choice([4, 6, 8])
    family = rng.choice(["lagrange", "spline", "spline"])
    m = 0 if family == "lagrange" else rng.choice([I // 2 - 1, I // 2 - 1, I // 2, 1])
    base = dict(kind=kind, N=N, family=family, I=I, m=m)
    cells = N ** 3
    if kind == "small":
        return dict(base, storage=rng.choice(["f64", "f32"]), np=_log_int(rng, 100, 30000),
                    scheme=rng.choice(["rk2", "ab2"]), dt=1e-3, steps=1)
    if kind == "step":
        storage = rng.choice(["f32", "f32", "f32", "f64", "bf16x2"])
        top = min(cells // 2, 1 << 17 if storage == "f64" else 1 << 21)
        return dict(base, storage=storage, np=_log_int(rng, max(1000, cells * 1.5e-3), max(2000, top)),
                    scheme=rng.choice(["rk2", "rk2", "ab2", "ab3", "ab4"]), dt=rng.choice([1e-3, 2.5e-3]),
                    steps=_log_int(rng, 1, 20 if storage != "f64" else 4))
    if kind == "coupled":
        return dict(base, storage=rng.choice(["f32", "f32", "bf16x2", "f64"]),
                    np=_log_int(rng, max(1000, cells * 1.5e-3), min(cells // 4, 1 << 20) + 1000),
                    scheme=rng.choice(["rk2", "ab2", "ab4"]), dt=2.5e-3, steps=1)
    if kind == "interp":
        deriv = rng.random() < 0.3
        C = 3 if deriv else rng.choice([1, 3, 3, 3, 12])
        storage = rng.choice(["f32", "f32", "f32", "bf16x2", "f64"])
        top = min(cells, (1 << 18) if storage == "f64" else (1 << 23) // (C // 3 if C > 3 else 1))
        return dict(base, storage=storage, np=_log_int(rng, max(1000, cells * 1.5e-3), max(2000, top)), C=C,
                    deriv=deriv, out="f64" if storage == "f64" else "f32")
    if kind == "batched":
        return dict(kind=kind, N=rng.choice([64, 128, 256, 512]), storage=rng.choice(["f32", "f32", "bf16x2"]),
                    nsets=rng.randint(2, 8), smallest=_log_int(rng, 10, 2000), largest=_log_int(rng, 20000, 1500000),
                    dt=2.5e-3, steps=rng.randint(1, 6))
    if kind == "adjoint":
        N = rng.choice([32, 64, 128, 256])
        return dict(base, N=N, storage=rng.choice(["f32", "f32", "bf16x2"]),
                    np=_log_int(rng, max(1000, N ** 3 * 1.5e-3), min(N ** 3 // 3, 1 << 21)), dt=2.5e-3,
                    steps=rng.randint(1, 5))
    return dict(kind="bin", N=N, np=_log_int(rng, 1000, 1 << 22))


def draw(rng):
    top = max(work(c)["flops"] for c in listed())
    while True:
        c = _draw_once(rng)
        if work(c)["flops"] <= 0.5 * top:
            return c


# --------------------------------------------------------------------------
# Inputs
# --------------------------------------------------------------------------
def _velocity(N, gen, grad):
    """u[3] (and du_k/dx_j as 3k + j) in float64: |u_hat| ~ k^(-11/6) for 1 <= |k| <= N / 3, divergence free."""
    dev = "cuda"
    kf = torch.fft.fftfreq(N, 1.0 / N, device=dev, dtype=torch.float64)
    kh = torch.fft.rfftfreq(N, 1.0 / N, device=dev, dtype=torch.float64)
    kvec = (kh[None, None, :], kf[None, :, None], kf[:, None, None])
    kk = kvec[0] ** 2 + kvec[1] ** 2 + kvec[2] ** 2
    kmax = N / 3.0
    ksafe = kk.clamp(min=1.0)
    amp = torch.where((kk >= 1.0) & (kk <= kmax * kmax), ksafe ** (-11.0 / 12.0), torch.zeros_like(kk))
    uh = [torch.complex(*(torch.randn(kk.shape, generator=gen, device=dev, dtype=torch.float64) for _ in range(2)))
          for _ in range(3)]
    kdotu = (kvec[0] * uh[0] + kvec[1] * uh[1] + kvec[2] * uh[2]) / ksafe
    uh = [(uh[a] - kvec[a] * kdotu) * amp for a in range(3)]
    u = [torch.fft.irfftn(x, s=(N, N, N)) for x in uh]
    s = 1.0 / math.sqrt(sum(float((x * x).mean()) for x in u) / 3.0)
    out = [x * s for x in u]
    if grad:
        out += [torch.fft.irfftn(1j * kvec[j] * uh[k], s=(N, N, N)) * s for k in range(3) for j in range(3)]
    return out


def _field(case, gen):
    N, C = case["N"], case.get("C", 3)
    dt = torch.float64 if case["storage"] == "f64" else torch.float32
    comps = _velocity(N, gen, C > 3)[:C]
    f = torch.empty((C, N, N, N), dtype=dt, device="cuda")
    for k, x in enumerate(comps):
        f[k] = x
    return f


def _positions(n, gen, spread):
    """Uniform tracers; spread > 0: some have moved out of the box by whole periods."""
    p = torch.rand((3, n), generator=gen, device="cuda", dtype=torch.float64) * TWO_PI
    if spread:
        p += torch.randint(-spread, spread + 1, (3, n), generator=gen, device="cuda").to(torch.float64) * TWO_PI
    return p


def _sets(case):
    """Sizes and kernels of a batched case: geometric sizes, I cycling 4, 6, 8, gradient outputs on odd sets."""
    k, a, b = case["nsets"], case["smallest"], case["largest"]
    out = []
    for i in range(k):
        n = int(round(a * (b / a) ** (i / max(k - 1, 1))))
        I = 4 + 2 * (i % 3)
        out.append(dict(np=n, I=I, m=I // 2 - 1, deriv=bool(i % 2)))
    return out


def _hist_rows(case):
    return {"rk2": 0, "ab2": 1, "ab3": 2, "ab4": 3}[case["scheme"]]


def _inputs(case, seed):
    """The seeded inputs of a case (prepare and exact both use them)."""
    gen = torch.Generator(device="cuda")
    gen.manual_seed(7919 * int(seed) + 17)
    kind, d = case["kind"], {}
    if kind == "bin":
        d["pos"] = _positions(case["np"], gen, 1)
        return d
    d["field"] = _field(case, gen)
    if kind == "batched":
        d["sets"] = []
        for s in _sets(case):
            rhs = 0.5 * torch.randn((3, s["np"]), generator=gen, device="cuda", dtype=torch.float32)
            d["sets"].append(dict(s, pos=_positions(s["np"], gen, 0), rhs=rhs))
        return d
    d["pos"] = _positions(case["np"], gen, 2 if kind in ("small", "coupled") or case.get("I") == 4 else 0)
    if kind in ("step", "small", "coupled") and _hist_rows(case):
        h = _hist_rows(case)
        d["rhs"] = 0.5 * torch.randn((h, 3, case["np"]), generator=gen, device="cuda", dtype=torch.float32)
    return d


def prepare(case, seed):
    s = _inputs(case, seed)
    s["case"] = case
    kind = case["kind"]
    if kind == "bin":
        s["tracker"] = trk.Tracker(case["N"])
    elif kind == "batched":
        s["tracker"] = trk.Tracker(case["N"], storage=STORAGE[case["storage"]])
        s["tracker"].set_field(s.pop("field"))
        for q in s["sets"]:
            q["out"] = torch.empty((9 if q["deriv"] else 3, q["np"]), device="cuda", dtype=torch.float32)
    else:
        s["tracker"] = trk.Tracker(case["N"], family=FAMILY[case["family"]], I=case["I"], m=case["m"],
                                   storage=STORAGE[case["storage"]])
        if kind == "adjoint":
            s["pos"] = s["pos"].float().requires_grad_(True)
            s["field"].requires_grad_(True)
        elif kind != "coupled":
            s["tracker"].set_field(s.pop("field"))
    torch.cuda.synchronize()
    return s


def _step(t, s, case):
    """From the kept initial state, so that every pass does the same steps."""
    pos = s["pos"].clone()
    if "rhs" not in s:
        t.advance(pos, case["dt"], case["steps"], SCHEME[case["scheme"]])
        return {"pos": pos}
    rhs = s["rhs"].clone()
    t.advance(pos, case["dt"], case["steps"], SCHEME[case["scheme"]], rhs=rhs, history_valid=rhs.shape[0])
    return {"pos": pos, "rhs": rhs}


def run(state):
    case, t = state["case"], state["tracker"]
    kind = case["kind"]
    if kind == "bin":
        keys, perm, offsets = t.bin(state["pos"])
        return {"keys": keys, "perm": perm, "offsets": offsets}
    if kind == "step":
        return _step(t, state, case)
    if kind == "small":
        u = t.interpolate(state["pos"], out_dtype=torch.float64 if case["storage"] == "f64" else torch.float32)
        return dict(_step(t, state, case), u=u)
    if kind == "coupled":
        t.set_field(state["field"])
        return _step(t, state, case)
    if kind == "interp":
        out = torch.float64 if case["out"] == "f64" else torch.float32
        return {"values": t.interpolate(state["pos"], out_dtype=out, deriv=case["deriv"])}
    if kind == "batched":
        sets = [dict(q, pos=q["pos"].clone(), rhs=q["rhs"].clone()) for q in state["sets"]]
        t.advance_batched(sets, case["dt"], case["steps"], history_valid=True)
        return [{"pos": q["pos"], "rhs": q["rhs"], "out": q["out"]} for q in sets]
    posT = advect(state["pos"].double(), state["field"], t, case["dt"], case["steps"])
    loss = (posT * posT).sum()
    gpos, gfield = torch.autograd.grad(loss, (state["pos"], state["field"]))
    return {"posT": posT.detach(), "grad_pos": gpos, "grad_field": gfield}


# --------------------------------------------------------------------------
# Work
# --------------------------------------------------------------------------
def _eval_flops(I, comps, grad=False):
    """Separable contraction of one stencil (x3, then x2, then x1) and its three sets of 1-D weights."""
    con = 2 * comps * (I ** 3 + I ** 2 + I)
    return (con * 2 if grad else con) + (2 if grad else 1) * 3 * I * 2 * I


def work(case):
    kind, n = case["kind"], case.get("np", 0)
    if kind == "bin":
        nb = (case["N"] // 8) ** 3
        return {"bytes": 24.0 * n + 8.0 * n + 4.0 * (nb + 1), "flops": 6.0 * n}
    N, C, esz = case["N"], case.get("C", 3), ESZ[case["storage"]]
    I = case.get("I", 8)
    fbytes = float(C) * N ** 3 * esz
    if kind == "batched":
        b, fl, nodes = 0.0, 0.0, 0.0
        for s in _sets(case):
            b += s["np"] * (48 + 24 + 4 * (9 if s["deriv"] else 3))
            fl += case["steps"] * s["np"] * (_eval_flops(s["I"], 3, s["deriv"]) + 30)
            nodes += float(s["np"]) * s["I"] ** 3
        return {"bytes": b + min(fbytes, nodes * 3 * esz), "flops": fl}
    seen = min(fbytes, float(n) * I ** 3 * C * esz)   # field values the stencils touch
    if kind == "interp":
        rows = 3 * C if case["deriv"] else C
        return {"bytes": seen + n * (24.0 + rows * (8 if case["out"] == "f64" else 4)),
                "flops": float(n) * _eval_flops(I, C, case["deriv"])}
    if kind == "adjoint":
        per = 2 * _eval_flops(I, 3) + 2 * _eval_flops(I, 3, True) + 2 * 2 * 3 * I ** 3 + 200
        return {"bytes": 2 * fbytes + n * (24.0 * 3), "flops": float(n) * case["steps"] * per}
    h = _hist_rows(case)
    evals = case["steps"] * (2 if case["scheme"] == "rk2" else 1)
    w = {"bytes": seen + n * (48.0 + 24.0 * h), "flops": float(n) * (evals * _eval_flops(I, C) + 30 * case["steps"])}
    if kind == "small":
        w = {"bytes": w["bytes"] + n * 24.0, "flops": w["flops"] + float(n) * _eval_flops(I, C)}
    if kind == "coupled":
        w["bytes"] = fbytes + n * (48.0 + 24.0 * h)
    return w


# --------------------------------------------------------------------------
# 64-bit values, in plain torch
# --------------------------------------------------------------------------
def _lagrange_poly(nodes, j):
    """Coefficients (ascending) of the Lagrange basis polynomial of nodes[j]."""
    c = [Fraction(1)]
    for i, x in enumerate(nodes):
        if i == j:
            continue
        den = Fraction(nodes[j] - x)
        c = [(c[k - 1] if k > 0 else 0) / den - (c[k] * x if k < len(c) else 0) / den for k in range(len(c) + 1)]
    return c


def _hermite(m):
    """h[end][order]: coefficients of the degree-(2m+1) polynomials on [0, 1] with one unit derivative at one end."""
    deg = 2 * m + 1
    rows = []
    for end in (0, 1):
        for o in range(m + 1):
            rows.append([Fraction(0) if k < o or (end == 0 and k > o) else
                         Fraction(math.factorial(k), math.factorial(k - o)) for k in range(deg + 1)])
    n = deg + 1
    a = [r + [Fraction(int(i == j)) for j in range(n)] for i, r in enumerate(rows)]
    for i in range(n):
        p = next(r for r in range(i, n) if a[r][i] != 0)
        a[i], a[p] = a[p], a[i]
        a[i] = [x / a[i][i] for x in a[i]]
        for r in range(n):
            if r != i and a[r][i] != 0:
                a[r] = [x - a[r][i] * y for x, y in zip(a[r], a[i])]
    inv = [[a[i][n + j] for j in range(n)] for i in range(n)]   # column j: the polynomial of condition j
    return [[[inv[k][e * (m + 1) + o] for k in range(n)] for o in range(m + 1)] for e in (0, 1)]


def _kernel(family, I, m):
    """Coefficients [I][deg+1] (ascending in t) of the weights of the nodes 1 - I/2 .. I/2."""
    nodes = list(range(1 - I // 2, I // 2 + 1))
    if family == "lagrange":
        rows = [_lagrange_poly(nodes, j) for j in range(I)]
    else:
        n = (I - 2) // 2
        cen = list(range(-n, n + 1))
        basis = [_lagrange_poly(cen, j) for j in range(2 * n + 1)]
        h = _hermite(m)
        rows = [[Fraction(0)] * (2 * m + 2) for _ in range(I)]
        for e in (0, 1):
            for o in range(m + 1):
                for j, q in zip(cen, basis):
                    d = (q[o] if o < len(q) else Fraction(0)) * math.factorial(o)   # derivative o at the node
                    row = rows[nodes.index(j + e)]
                    for k in range(2 * m + 2):
                        row[k] += d * h[e][o][k]
    return torch.tensor([[float(x) for x in r] for r in rows], dtype=torch.float64, device="cuda")


def _poly(c, t):
    w = c[:, -1][None, :].expand(t.shape[0], -1)
    for k in range(c.shape[1] - 2, -1, -1):
        w = w * t[:, None] + c[:, k][None, :]
    return w


def _stencil(x, N, I, c, dc):
    """Node indices [p, I^3] and 1-D weights (and derivatives per unit length) of positions x[3][p]."""
    g = x * (N / TWO_PI)
    cell = torch.floor(g)
    t = g - cell
    off = torch.arange(1 - I // 2, I // 2 + 1, device="cuda")
    ix = [((cell[a].long()[:, None] + off[None, :]) % N) for a in range(3)]
    idx = (ix[2][:, :, None, None] * N + ix[1][:, None, :, None]) * N + ix[0][:, None, None, :]
    w = [_poly(c, t[a]) for a in range(3)]
    dw = [_poly(dc, t[a]) * (N / TWO_PI) for a in range(3)]
    return idx.reshape(x.shape[1], -1), w, dw


def _contract(v, w1, w2, w3):
    return ((((v * w1[:, None, None, :]).sum(-1) * w2[:, None, :]).sum(-1)) * w3).sum(-1)


class _Exact:
    def __init__(self, case, field, I=None, family=None, m=None):
        self.N, self.I = case["N"], I or case["I"]
        self.c = _kernel(family or case["family"], self.I, case["m"] if m is None else m)
        self.dc = self.c[:, 1:] * torch.arange(1, self.c.shape[1], device="cuda", dtype=torch.float64)
        self.f = field.detach().double().reshape(field.shape[0], -1)
        self.chunk = max(1, (1 << 25) // self.I ** 3)

    def chunks(self, n):
        return [(a, min(n, a + self.chunk)) for a in range(0, n, self.chunk)]

    def values(self, x, grad=False):
        n, C = x.shape[1], self.f.shape[0]
        out = torch.empty((C, n), dtype=torch.float64, device="cuda")
        g = torch.empty((3 * C, n), dtype=torch.float64, device="cuda") if grad else None
        for a, b in self.chunks(n):
            idx, w, dw = _stencil(x[:, a:b], self.N, self.I, self.c, self.dc)
            for k in range(C):
                v = self.f[k][idx].reshape(b - a, self.I, self.I, self.I)
                out[k, a:b] = _contract(v, w[0], w[1], w[2])
                if grad:
                    for j in range(3):
                        q = [dw[i] if i == j else w[i] for i in range(3)]
                        g[3 * k + j, a:b] = _contract(v, *q)
        return (out, g) if grad else out

    def rk2(self, x, dt):
        k1 = self.values(x)
        return x + (0.5 * dt) * (k1 + self.values(x + dt * k1))

    def scatter(self, g, x, mu):
        """g[k][node] += weight * mu[k]"""
        for a, b in self.chunks(x.shape[1]):
            idx, w, _ = _stencil(x[:, a:b], self.N, self.I, self.c, self.dc)
            W = (w[2][:, :, None, None] * w[1][:, None, :, None] * w[0][:, None, None, :]).reshape(b - a, -1)
            for k in range(3):
                g[k].index_add_(0, idx.reshape(-1), (W * mu[k, a:b, None]).reshape(-1))


_BETA = [[1.0], [1.5, -0.5], [23 / 12, -16 / 12, 5 / 12], [55 / 24, -59 / 24, 37 / 24, -9 / 24]]


def _advance_exact(E, case, x, rhs):
    x = x.clone()
    if rhs is None:
        for _ in range(case["steps"]):
            x = E.rk2(x, case["dt"])
        return {"pos": x}
    hist = [rhs[i].double() for i in range(rhs.shape[0])]
    for _ in range(case["steps"]):
        us = [E.values(x)] + hist
        x = x + case["dt"] * sum(b * u for b, u in zip(_BETA[len(hist)], us))
        hist = us[:len(hist)]
    return {"pos": x, "rhs": torch.stack(hist)}


def exact(case, seed):
    kind = case["kind"]
    if kind == "bin":
        return None                      # whole numbers
    d = _inputs(case, seed)
    with torch.no_grad():
        if kind == "batched":
            out = []
            for s in d["sets"]:
                E = _Exact(case, d["field"], I=s["I"], family="spline", m=s["m"])
                x, h = s["pos"].clone(), s["rhs"].double()
                for _ in range(case["steps"]):
                    r = E.values(x, s["deriv"])
                    u, o = r if s["deriv"] else (r, r)
                    x = x + case["dt"] * (1.5 * u - 0.5 * h)
                    h = u
                out.append({"pos": x, "rhs": h, "out": o})
            return out
        E = _Exact(case, d["field"])
        if kind == "interp":
            return {"values": E.values(d["pos"], True)[1] if case["deriv"] else E.values(d["pos"])}
        if kind in ("step", "coupled", "small"):
            out = _advance_exact(E, case, d["pos"], d.get("rhs"))
            if kind == "small":
                out["u"] = E.values(d["pos"])
            return out
        xs, dt = [d["pos"].float().double()], case["dt"]
        for _ in range(case["steps"]):
            xs.append(E.rk2(xs[-1], dt))
        lam = 2.0 * xs[-1]
        g = torch.zeros_like(E.f)
        for x in reversed(xs[:-1]):
            u, J = E.values(x, True)
            xs2 = x + dt * u
            Js = E.values(xs2, True)[1]
            ls = 0.5 * dt * (Js.reshape(3, 3, -1) * lam[:, None, :]).sum(0)
            mu = 0.5 * dt * lam + dt * ls
            E.scatter(g, x, mu)
            E.scatter(g, xs2, 0.5 * dt * lam)
            lam = lam + ls + (J.reshape(3, 3, -1) * mu[:, None, :]).sum(0)
        return {"posT": xs[-1], "grad_pos": lam, "grad_field": g.reshape(d["field"].shape)}
