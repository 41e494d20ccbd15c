"""What is measured: the work a user has the library do, through its public entry points.

A case is a dict of plain values.  ``kind`` names the call:

  monitor      iterations one by one, D_TPL read after each (the convergence trace of a study)
  reconstruct  one whole solve from host counts to host maps (osscir_reconstruct)
  iterate      counts already on the device: MOCCA iterations, then the solver state
  forward      X x of four channels           backproject  X^T rf of four channels
  simulate     expected counts of maps, then their seeded Poisson noise (making study data)
  batch        several different solves advanced together
  new          a new problem (geometry, spectra) from its creation to its first iterates

``exact`` restates the method in plain torch FP64 (Siddon lengths slab by slab, the
counts model, the eigen-clipped curvature, the dual prox, the pixel step).
"""
from __future__ import annotations

import functools
import math

import numpy as np
import torch

import paper_1801_06263_gb300 as pkg
from paper_1801_06263_gb300 import _lib, inputs

# The fields of a solve, with the values of the named workloads.
BASE = {"n": 256, "views": 512, "bins": 512, "photons": 1e5, "windows": 4, "model": 0, "spc": 0,
        "exp": 0, "box": 0, "inner": 1, "iters": 10}


def _case(kind, name=None, **kw):
    c = dict(BASE, kind=kind, **kw)
    if name is not None:
        c["name"] = name
    return c


def listed():
    return [
        # The smallest calls: a 64x64 study solve (small_64) stepped one iteration at a time
        # with its D_TPL read back after each, as a convergence plot is made.
        _case("monitor", "monitor_64", n=64, views=128, bins=128, iters=20),
        # The same small solve whole, from pinned host counts to host maps: 200 short iterations.
        _case("reconstruct", "reconstruct_64", n=64, views=128, bins=128, iters=200),
        # The headline workload (medium_256).
        _case("iterate", "iterate_256"),
        # The largest workload (large_512).
        _case("iterate", "iterate_512", n=512, views=1024, bins=1024, photons=1e6, iters=4),
        # Ragged sizes (no multiple of a warp, tile or group) with nonnegative maps.
        _case("iterate", "ragged_389_nonneg", n=389, views=541, bins=397, photons=3e4, box=1),
        # Five ideal-layout windows with the separable curvature, the reading that gives the
        # paper's ordering of the preconditioners.
        _case("iterate", "five_windows_256", windows=5, model=3),
        # Nested inner/outer iterations at an uneven size.
        _case("iterate", "nested_300", n=300, views=251, bins=306, inner=4, iters=12),
        # The projector pair on its own, for a caller's own algorithm.
        _case("forward", "forward_256"),
        _case("backproject", "backproject_256"),
        # Making the data of a study at the largest size.
        _case("simulate", "simulate_512", n=512, views=1024, bins=1024, photons=1e6),
        # Twelve mixed reconstructions (sizes, doses and view counts of the batched workload).
        _case("batch", "batch_12", solves=12, recipe=4000, iters=2),
        # A new scanner or protocol: creation, tables and the first iterations.
        _case("new", "new_256"),
    ]


def _log_int(rng, lo, hi):
    return int(round(math.exp(rng.uniform(math.log(lo), math.log(hi)))))


def draw(rng):
    kind = rng.choice(["monitor", "reconstruct", "iterate", "iterate", "iterate", "iterate", "forward",
                       "backproject", "simulate", "batch", "new"])
    if kind == "batch":
        return _case("batch", solves=rng.randint(3, 12), recipe=rng.randint(4001, 9000), iters=rng.choice([1, 2]))
    hi = 96 if kind in ("monitor", "reconstruct") else 384 if kind == "new" else 512
    n = _log_int(rng, 16, hi)
    views = max(24, int(n * rng.uniform(0.6, 2.0)))
    bins = max(24, int(n * rng.uniform(0.8, 2.0)))
    c = _case(kind, n=n, views=views, bins=bins, photons=float(round(10.0 ** rng.uniform(4.0, 6.0))))
    if kind == "monitor":
        c["iters"] = rng.randint(5, 20)
    elif kind == "reconstruct":
        c["iters"] = rng.randint(40, 200)
    elif kind == "iterate":
        c["iters"] = rng.randint(1, 4) if n > 300 else rng.randint(2, 10)
        c["model"] = rng.choice([0, 0, 0, 1, 2, 3])
        c["spc"] = rng.choice([0, 0, 0, 1, 2])
        c["exp"] = rng.choice([0, 0, 0, 1])
        c["box"] = rng.choice([0, 0, 1]) if c["spc"] == 0 else 0
        c["windows"] = rng.choice([4, 4, 4, 5])
        if c["windows"] == 4:
            c["inner"] = rng.choice([1, 1, 1, 2, 4])
    return c


# --------------------------------------------------------------------------- inputs

def _geom(c):
    return inputs.make_geometry(c["n"], 0.5, c["views"], c["bins"])


@functools.lru_cache(maxsize=64)
def _spectra(bins, photons, windows):
    """The scanner's spectral response (fixed for a scanner, not part of a data set)."""
    return inputs.make_spectra(bins, photons, n_windows=windows)


def _lam(c):
    """The stable step ratio of the size and dose; the comparison preconditioner's own is far larger."""
    lam = inputs.step_ratio(c["n"], c["photons"])
    return lam if c["spc"] == 0 else 0.1 * lam


def _ellipses(n, seed):
    """A body of PMMA with Al and Gd inserts at seeded places: rows (cx, cy, ax, ay, dPMMA, dAl, dGd)."""
    rng = np.random.default_rng(seed)
    nh = 0.5 * n
    ax, ay = rng.uniform(0.36, 0.43) * nh, rng.uniform(0.30, 0.38) * nh
    rows = [(0.0, 0.0, ax, ay, 1.0, 0.0, 0.0)]
    for i in range(10):
        t, rad, r = 2 * math.pi * (i + rng.uniform(0.1, 0.9)) / 10, rng.uniform(0.45, 0.7), rng.uniform(0.03, 0.055) * nh
        al = i % 5 < 2
        rows.append((rad * ax * math.cos(t), rad * ay * math.sin(t), r, r, -1.0 if al else 0.0, 1.0 if al else 0.0,
                     0.0 if al else float(rng.uniform(0.001, 0.02))))
    return rows


def _rays(g):
    """Foot points and unit directions [L, 2] (FP64, device) of a geometry's rays."""
    v = torch.arange(g.n_views, dtype=torch.float64, device="cuda")
    th = (g.start_deg + v * g.arc_deg / g.n_views) * math.pi / 180.0
    u = (torch.arange(g.n_bins, dtype=torch.float64, device="cuda") - 0.5 * (g.n_bins - 1)) * g.bin_mm
    c, s = torch.cos(th)[:, None], torch.sin(th)[:, None]
    back = g.sid_mm - g.sdd_mm
    S = torch.stack([(g.sid_mm * c).expand(-1, g.n_bins), (g.sid_mm * s).expand(-1, g.n_bins)], -1)
    D = torch.stack([back * c - u * s, back * s + u * c], -1)
    d = D - S
    d = d / d.norm(dim=-1, keepdim=True)
    B = S - (S * d).sum(-1, keepdim=True) * d
    return B.reshape(-1, 2), d.reshape(-1, 2)


def _line_integrals(g, rows):
    """Closed-form line integrals [L, 3] of the ellipses."""
    B, d = _rays(g)
    out = torch.zeros((B.shape[0], 3), dtype=torch.float64, device="cuda")
    for cx, cy, ax, ay, *val in rows:
        sc = torch.tensor([1.0 / ax, 1.0 / ay], dtype=torch.float64, device="cuda")
        o = (B - torch.tensor([cx, cy], dtype=torch.float64, device="cuda")) * sc
        q = d * sc
        a, b, k = (q * q).sum(-1), (o * q).sum(-1), (o * o).sum(-1) - 1.0
        chord = 2.0 * torch.sqrt(torch.clamp(b * b - a * k, min=0.0)) / a
        out += chord[:, None] * torch.tensor(val, dtype=torch.float64, device="cuda")
    return out


def _counts(c, seed):
    """Measured counts [L, WS] (float32, device) of a seeded object: exp model of its exact line
    integrals and Poisson noise, made here so that they do not depend on the library."""
    g, sp, W = _geom(c), _spectra(c["bins"], c["photons"], c["windows"]), c["windows"]
    li = _line_integrals(g, _ellipses(c["n"], seed)).reshape(g.n_views, g.n_bins, 3)
    mu = torch.as_tensor(sp.mu, device="cuda")
    s = torch.as_tensor(sp.s, device="cuda")
    N = torch.as_tensor(sp.N, device="cuda")
    out = torch.zeros((g.n_views, g.n_bins, _lib.window_stride(W)), dtype=torch.float32, device="cuda")
    gen = torch.Generator(device="cuda").manual_seed(seed)
    for v in range(0, g.n_views, 128):
        e = torch.exp(-(li[v:v + 128] @ mu))                                  # [v, b, i]
        chat = N * torch.bmm(e.transpose(0, 1), s).transpose(0, 1)             # [v, b, w]
        out[v:v + 128, :, :W] = torch.poisson(chat, generator=gen).float()
    return out.reshape(g.n_rays, -1)


def _maps(c, seed):
    """Smooth random material maps [P, 4] (float32, device) in the range of real ones."""
    n = c["n"]
    gen = torch.Generator(device="cuda").manual_seed(seed)
    y, x = torch.meshgrid(torch.linspace(-1, 1, n, device="cuda"), torch.linspace(-1, 1, n, device="cuda"), indexing="ij")
    body = ((x / 0.84) ** 2 + (y / 0.68) ** 2 <= 1).float()
    m = torch.rand((n, n, 4), device="cuda", generator=gen) * 0.1 - 0.05
    m[..., 0] += body
    m[..., 1] += body * 0.2 * torch.rand((1,), device="cuda", generator=gen)
    m[..., 2] = body * 0.01 * torch.rand((n, n), device="cuda", generator=gen)
    m[..., 3] = torch.rand((n, n), device="cuda", generator=gen)
    return m.reshape(n * n, 4).contiguous()


_BOX = ((0.0, 0.0, 0.0), (float("inf"),) * 3)


def _recon(c):
    return pkg.Reconstructor(_geom(c), _spectra(c["bins"], c["photons"], c["windows"]), _lam(c), model=c["model"],
                             box=_BOX if c["box"] else None, spc=c["spc"], counts_model=c["exp"], inner=c["inner"])


def _members(c):
    """The solves of a batch: the batched workload's sizes, views and doses."""
    rng = np.random.default_rng(c["recipe"])
    out = []
    for _ in range(c["solves"]):
        n, views = int(rng.choice([128, 192, 256, 384, 512])), int(rng.integers(90, 721))
        out.append(dict(BASE, kind="iterate", n=n, views=views, bins=views, photons=float(10.0 ** rng.uniform(4.0, 6.0)),
                        iters=c["iters"]))
    return out


# --------------------------------------------------------------------------- preparing and running

def prepare(case, seed):
    c, kind = dict(case), case["kind"]
    st = {"case": c}
    if kind == "batch":
        st["recons"] = [_recon(m) for m in _members(c)]
        st["counts"] = [_counts(m, 1000 * seed + i) for i, m in enumerate(_members(c))]
        st["batch"] = pkg.Batch(st["recons"])
        return st
    if kind == "new":
        _spectra(c["bins"], c["photons"], c["windows"])
        st["c"] = _counts(c, seed)
        return st
    st["R"] = _recon(c)
    if kind == "forward":
        st["x"] = _maps(c, seed)
    elif kind == "backproject":
        gen = torch.Generator(device="cuda").manual_seed(seed)
        st["rf"] = torch.randn((c["views"] * c["bins"], 4), device="cuda", generator=gen)
    elif kind == "simulate":
        st["x"] = _maps(c, seed)
        st["seed"] = int(seed)
    elif kind == "reconstruct":
        st["c"] = _counts(c, seed).cpu().pin_memory()
        st["out"] = torch.zeros((c["n"] ** 2, 4), dtype=torch.float32).pin_memory()
    else:
        st["c"] = _counts(c, seed)
    return st


def run(state):
    c = state["case"]
    kind = c["kind"]
    if kind == "forward":
        return state["R"].forward(state["x"])
    if kind == "backproject":
        return state["R"].backproject(state["rf"])
    if kind == "simulate":
        chat = state["R"].simulate(state["x"])
        return {"chat": chat, "counts": _lib.osscir_poisson_noise(chat, state["seed"])}
    if kind == "reconstruct":
        _lib.osscir_reconstruct(state["R"].handle, state["c"], c["iters"], state["out"])
        return {"maps": state["out"]}
    if kind == "monitor":
        R, trace = state["R"], []
        R.set_counts(state["c"])
        for _ in range(c["iters"]):
            R.step(1)
            trace.append(R.dtpl(1))
        return {"maps": R.maps(), "trace": trace}
    if kind == "batch":
        for R, cnt in zip(state["recons"], state["counts"]):
            R.set_counts(cnt)
        state["batch"].step(c["iters"])
        return [R.maps() for R in state["recons"]]
    if kind == "new":
        R = _recon(c)
        R.set_counts(state["c"])
        R.step(c["iters"])
        maps = R.maps()
        R.close()
        return {"maps": maps}
    R = state["R"]
    R.set_counts(state["c"])
    R.step(c["iters"])
    x, xbar, y, _ = R.get_state()
    return {"x": x, "xbar": xbar, "y": y}


# --------------------------------------------------------------------------- the least work

def _solve_work(c):
    """Bytes (counts in, maps, extrapolation and duals out) and operations (three channels forward,
    nine back, the counts model with its two derivatives) of c["iters"] iterations."""
    L, P, W, nE = c["views"] * c["bins"], c["n"] ** 2, c["windows"], 101
    pairs = 0.83 * L * c["n"]
    outer = -(-c["iters"] // c["inner"])
    return {"bytes": 4.0 * (2 * W * L + 6 * P),
            "flops": c["iters"] * 24.0 * pairs + outer * 2.0 * L * nE * (3 + 10 * W)}


def work(case):
    c, kind = case, case["kind"]
    L, P = c["views"] * c["bins"], c["n"] ** 2
    if kind == "batch":
        ws = [_solve_work(m) for m in _members(c)]
        return {"bytes": sum(w["bytes"] for w in ws), "flops": sum(w["flops"] for w in ws)}
    if kind in ("forward", "backproject"):
        return {"bytes": 16.0 * (L + P), "flops": 8.0 * 0.83 * L * c["n"]}
    if kind == "simulate":
        return {"bytes": 12.0 * P + 32.0 * L, "flops": 6.0 * 0.83 * L * c["n"] + 2.0 * L * 101 * 7}
    return _solve_work(c)


# --------------------------------------------------------------------------- FP64 restatement

def _pairs(g, B, d):
    """Pixels [R, n, 2] and lengths of rays (B, d): along the ray's dominant axis every slab of
    pixels is crossed once and touches at most two of them."""
    n, h, x0 = g.n, g.pixel_mm, -0.5 * g.n * g.pixel_mm
    rows = d[:, 1].abs() >= d[:, 0].abs()
    bM, bm = torch.where(rows, B[:, 1], B[:, 0]), torch.where(rows, B[:, 0], B[:, 1])
    dM, dm = torch.where(rows, d[:, 1], d[:, 0]), torch.where(rows, d[:, 0], d[:, 1])
    planes = x0 + torch.arange(n + 1, dtype=torch.float64, device=B.device) * h
    t = (planes[None] - bM[:, None]) / dM[:, None]
    m = (bm[:, None] + t * dm[:, None] - x0) / h             # minor position at the planes, in pixels
    m0, m1, t0, t1 = m[:, :-1], m[:, 1:], t[:, :-1], t[:, 1:]
    lo, hi = torch.minimum(m0, m1), torch.maximum(m0, m1)
    ia, ib = torch.floor(lo), torch.floor(hi)
    full = (t1 - t0).abs()
    cut = torch.where(ib > ia, (ib - lo) / torch.where(ib > ia, hi - lo, torch.ones_like(hi)), torch.ones_like(hi))
    ln = torch.stack([full * cut, full * (1.0 - cut)], -1)
    mi = torch.stack([ia, ib], -1)
    ok = (mi >= 0) & (mi < n) & (ln > 1e-9 * h)
    j = torch.arange(n, device=B.device)[None, :, None]
    mi = mi.clamp(0, n - 1).long()
    k = torch.where(rows[:, None, None], j * n + mi, mi * n + j)
    return k, torch.where(ok, ln, torch.zeros_like(ln))


def _chunks(g):
    B, d = _rays(g)
    step = max(1, 24_000_000 // (2 * g.n))
    for l in range(0, g.n_rays, step):
        yield slice(l, min(g.n_rays, l + step)), *_pairs(g, B[l:l + step], d[l:l + step])


def _X(g, f):
    out = torch.empty((g.n_rays, f.shape[1]), dtype=torch.float64, device="cuda")
    for sl, k, w in _chunks(g):
        for ch in range(f.shape[1]):
            out[sl, ch] = (f[:, ch][k] * w).sum((1, 2))
    return out


def _Xt(g, y):
    out = torch.zeros((y.shape[1], g.n_pixels), dtype=torch.float64, device="cuda")
    for sl, k, w in _chunks(g):
        k = k.reshape(-1)
        for ch in range(y.shape[1]):
            out[ch].index_add_(0, k, (w * y[sl, ch][:, None, None]).reshape(-1))
    return out.T.contiguous()


def _clip(H):
    """Negative eigenvalues of the symmetric H [L, 3, 3] removed (cyclic Jacobi)."""
    a = H.clone()
    V = torch.eye(3, dtype=H.dtype, device=H.device).expand_as(H).clone()
    for _ in range(7):
        for p, q in ((0, 1), (0, 2), (1, 2)):
            apq = a[:, p, q]
            zero = apq == 0
            tau = (a[:, q, q] - a[:, p, p]) / torch.where(zero, torch.ones_like(apq), 2 * apq)
            t = torch.where(tau >= 0, 1.0, -1.0) / (tau.abs() + torch.sqrt(1 + tau * tau))
            t = torch.where(zero, torch.zeros_like(t), t)
            cs = torch.rsqrt(1 + t * t)[:, None]
            sn = t[:, None] * cs
            cp, cq = a[:, :, p].clone(), a[:, :, q].clone()
            a[:, :, p], a[:, :, q] = cs * cp - sn * cq, sn * cp + cs * cq
            rp, rq = a[:, p, :].clone(), a[:, q, :].clone()
            a[:, p, :], a[:, q, :] = cs * rp - sn * rq, sn * rp + cs * rq
            vp, vq = V[:, :, p].clone(), V[:, :, q].clone()
            V[:, :, p], V[:, :, q] = cs * vp - sn * vq, sn * vp + cs * vq
    lam = torch.diagonal(a, dim1=1, dim2=2).clamp(min=0)
    return (V * lam[:, None, :]) @ V.transpose(1, 2)


def _spd_solve(M, b):
    """x of M x = b for positive definite M [L, k, k], b [L, k] (elimination)."""
    M, b, k = M.clone(), b.clone(), M.shape[1]
    for c in range(k):
        for r in range(c + 1, k):
            f = M[:, r, c] / M[:, c, c]
            M[:, r, c:] -= f[:, None] * M[:, c, c:].clone()
            b[:, r] -= f * b[:, c]
    x = torch.zeros_like(b)
    for r in range(k - 1, -1, -1):
        x[:, r] = (b[:, r] - (M[:, r, r + 1:] * x[:, r + 1:]).sum(-1)) / M[:, r, r]
    return x


class _Model:
    """The spectral model of a solve in FP64, from the float32 inputs the library takes."""

    def __init__(self, c):
        sp = _spectra(c["bins"], c["photons"], c["windows"])
        f32 = lambda a: torch.as_tensor(np.asarray(a, dtype=np.float32).astype(np.float64), device="cuda")
        self.c, self.s, self.N, self.mu = c, f32(sp.s), f32(sp.N), f32(sp.mu)
        if c["spc"] == 2:   # curves orthonormal over the energy grid: M = (mu mu^T)^(-1/2)
            w, V = torch.linalg.eigh(self.mu @ self.mu.T)
            self.M = V @ torch.diag(w.rsqrt()) @ V.T
            self.mu_in, self.mu = self.mu, (self.M @ self.mu).float().double()

    def sexp(self, p, expm):
        e = torch.exp(-p)
        if expm:
            return e, e, e
        neg = p < 0
        return (torch.where(neg, 1 - p, e), torch.where(neg, torch.ones_like(e), e),
                torch.where(neg, torch.zeros_like(e), e))

    def counts(self, li, mu):
        nb = self.c["bins"]
        out = []
        for li_v in li.reshape(-1, nb, 3).split(64):
            e0 = self.sexp(li_v @ mu, self.c["exp"])[0]
            out.append(self.N * torch.bmm(e0.transpose(0, 1), self.s).transpose(0, 1))
        return torch.cat(out).reshape(-1, self.c["windows"])

    def terms(self, li, cnt):
        """chat, alpha [L, W, 3] and the Hessian [L, 3, 3] at the line integrals."""
        nb, W = self.c["bins"], self.c["windows"]
        mm = torch.einsum("mi,ni->imn", self.mu, self.mu).reshape(-1, 9)
        ch, al, Hs = [], [], []
        for li_v, c_v in zip(li.reshape(-1, nb, 3).split(64), cnt.reshape(-1, nb, W).split(64)):
            e0, e1, e2 = self.sexp(li_v @ self.mu, self.c["exp"])
            D = torch.bmm(e0.transpose(0, 1), self.s).transpose(0, 1)
            a = torch.stack([torch.bmm((e1 * self.mu[m]).transpose(0, 1), self.s).transpose(0, 1) / D for m in range(3)], -1)
            chat = self.N * D
            beta = e2 * torch.bmm(((c_v - chat) / D).transpose(0, 1), self.s.transpose(1, 2)).transpose(0, 1)
            H = -(beta @ mm).reshape(*beta.shape[:2], 3, 3)
            if self.c["model"] == 2:
                H = torch.zeros_like(H)
            H = H + torch.einsum("vbw,vbwm,vbwn->vbmn", c_v, a, a)
            ch.append(chat.reshape(-1, W))
            al.append(a.reshape(-1, W, 3))
            Hs.append(H.reshape(-1, 3, 3))
        return torch.cat(ch), torch.cat(al), torch.cat(Hs)


def _dtpl(chat, c):
    return float(torch.where(c > 0, chat - c - c * torch.log(chat / torch.where(c > 0, c, torch.ones_like(c))), chat).sum())


def _box_step(Q, t):
    """argmin over x >= 0 of (x - t)^T Q (x - t): the feasible candidate of least objective."""
    best = torch.full_like(t[:, 0], math.inf)
    out = t.clamp(min=0)
    for code in range(8):
        fr = [m for m in range(3) if not code >> m & 1]
        fx = [m for m in range(3) if code >> m & 1]
        x = torch.zeros_like(t)
        if fr:
            rhs = (Q[:, fr][:, :, fx] * t[:, None, fx]).sum(-1) if fx else torch.zeros_like(t[:, fr])
            x[:, fr] = t[:, fr] + _spd_solve(Q[:, fr][:, :, fr], rhs)
        ok = (x >= -1e-12 * (1 + x.abs())).all(-1)
        x = x.clamp(min=0)
        obj = torch.einsum("li,lij,lj->l", x - t, Q, x - t)
        take = ok & (obj < best)
        best = torch.where(take, obj, best)
        out = torch.where(take[:, None], x, out)
    return out


def _mocca(c, cnt):
    """c["iters"] iterations from zero: x, xbar, y, D_TPL at each outer expansion point."""
    g, S = _geom(c), _Model(c)
    W, lam, blk = c["windows"], float(np.float32(_lam(c))), c["spc"] == 0
    cnt = cnt[:, :W].double()
    dev = dict(dtype=torch.float64, device="cuda")
    x, xbar, y = torch.zeros((g.n_pixels, 3), **dev), torch.zeros((g.n_pixels, 3), **dev), torch.zeros((g.n_rays, W), **dev)
    X1 = _X(g, torch.ones((g.n_pixels, 1), **dev))
    hit = (X1[:, 0] > 0)
    trace = []
    for it in range(c["iters"]):
        li = _X(g, xbar)
        if it % c["inner"] == 0:
            chat, al, H = S.terms(li, cnt)
            trace.append(_dtpl(chat, cnt))
            r = cnt - chat
            nw = al.norm(dim=-1) if blk else al.abs().sum(-1)
            sinv = torch.where(hit[:, None], lam * X1 * nw, torch.ones_like(nw))
            if c["model"] in (0, 2):
                Hp = _clip(H) if c["model"] == 0 else H
                A = al.transpose(1, 2) @ al
                G = torch.stack([_spd_solve(A, al[:, w]) for w in range(W)], -1)
                Wm = G.transpose(1, 2) @ Hp @ G
            elif c["model"] == 3:
                Wm = torch.diag_embed(cnt)
            else:
                Wm = torch.zeros((g.n_rays, W, W), **dev)
            Mx = Wm + torch.diag_embed(1 / sinv)
            if blk:
                Sm = torch.einsum("lwm,lwn,lw->lmn", al, al, 1 / nw)
            else:
                Sm = torch.diag_embed(al.abs().sum(1))
            P = _Xt(g, Sm.reshape(-1, 9)[:, [0, 1, 2, 4, 5, 8]])
            Tinv = P[:, [0, 1, 2, 1, 3, 4, 2, 4, 5]].reshape(-1, 3, 3) / lam
            tr = torch.diagonal(Tinv, dim1=1, dim2=2).sum(-1)
            seen = tr > 0
            Tinv = torch.where(seen[:, None, None], Tinv + torch.diag_embed((1e-12 * tr)[:, None].expand(-1, 3)),
                               torch.eye(3, **dev))
            li0 = li
        u = y + torch.einsum("lwm,lm->lw", al, li - li0) / sinv
        yn = u - _spd_solve(Mx, u - r) / sinv
        y = torch.where(hit[:, None], yn, y)
        v = _Xt(g, torch.einsum("lwm,lw->lm", al, y))
        t = x - _spd_solve(Tinv, v)
        if c["box"]:
            out = (t < 0).any(-1)
            t[out] = _box_step(Tinv[out], t[out])
        xn = torch.where(seen[:, None], t, x)
        xbar, x = 2 * xn - x, xn
    return S, x, xbar, y, trace


def _pad(t, k):
    return torch.nn.functional.pad(t, (0, k - t.shape[1]))


def _exact_maps(c, cnt):
    S, x, *_ = _mocca(c, cnt)
    return _pad(x @ S.M.T if c["spc"] == 2 else x, 4)


def exact(case, seed):
    c, kind = dict(case), case["kind"]
    g = _geom(c)
    if kind == "forward":
        return _X(g, _maps(c, seed).double())
    if kind == "backproject":
        gen = torch.Generator(device="cuda").manual_seed(seed)
        return _Xt(g, torch.randn((g.n_rays, 4), device="cuda", generator=gen).double())
    if kind == "simulate":
        S = _Model(c)
        return {"chat": _pad(S.counts(_X(g, _maps(c, seed)[:, :3].double()), S.mu), 4), "counts": None}
    if kind == "batch":
        return [_exact_maps(m, _counts(m, 1000 * seed + i)) for i, m in enumerate(_members(c))]
    if kind in ("new", "reconstruct"):
        return {"maps": _exact_maps(c, _counts(c, seed))}
    S, x, xbar, y, trace = _mocca(c, _counts(c, seed))
    if kind == "monitor":
        return {"maps": _pad(x, 4), "trace": trace}
    return {"x": _pad(x, 4), "xbar": _pad(xbar, 4), "y": _pad(y, _lib.window_stride(c["windows"]))}
