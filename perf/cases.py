"""The work that users of this library have it do, as measurable cases.

A case is one call (or the fixed sequence of calls that belongs to one step of a
user's program) through the public Python API, on media of the kinds the library
is written for: stratified scattering atmospheres, log-normal turbulent boxes,
multi-frequency atmospheres and 2D planes.  ``kind`` says which calls:

* ``formal``   rt.Grid.formal_solve of a given S on a standing medium (J, Lambda*):
               one Lambda operator application, as an outer solver asks for it.
* ``noalloc``  rt.formal_solve_noalloc: the same without a grid, for a host code
               that keeps the device memory in its own pool.
* ``medium``   rt.Grid.set_opacity_source of a new medium, and one formal solution.
* ``step``     the radiation step of a time-dependent run: the new medium, a few
               ALI iterations from the previous S, then J, H and Q for the gas
               (the paper's runs take one to five iterations a step).
* ``solve``    the whole job: medium, ALI from S = B until converged (or out of
               iterations), S, and the moments that a VET and the gas need.
* ``many``     rt.ali_solve_many: several standing problems of different sizes
               solved together.

A mixed grid (float32 sweeps) returns numbers of float32 accuracy; the programs
that choose it keep them in float32, as ``run`` does here.  FP64 grids' results
stay in float64.
"""
import math

import numpy as np
import torch

from paper_1201_2222_gb300 import rt

P, V, T = rt.PERIODIC, rt.VACUUM, rt.THERMAL
DEV = "cuda"
F64 = torch.float64


def _case(kind, nx, ny, nz, n_mu, prec, medium, nf=1, eps=1e-2, tol=1e-6, max_iter=1, interp="linear"):
    return dict(kind=kind, nx=nx, ny=ny, nz=nz, n_mu=n_mu, prec=prec, medium=medium, nf=nf, eps=eps, tol=tol,
                max_iter=max_iter, interp=interp)


def listed():
    def c(name, *a, **k):
        return dict(_case(*a, **k), name=name)

    return [
        # a small Lambda application inside somebody else's time loop, no allocation allowed: latency
        c("noalloc_24_mixed", "noalloc", 24, 24, 24, 4, "mixed", "atmosphere"),
        # the FP64 formal solution of the 32^3 atmosphere with Lambda*: latency, launches
        c("formal_32_fp64", "formal", 32, 32, 32, 4, "fp64", "atmosphere"),
        # one radiation step of a small time-dependent box, warm-started
        c("step_48_mixed", "step", 48, 48, 48, 6, "mixed", "box", max_iter=5),
        # the paper's scattering atmosphere to convergence, everything in FP64
        c("solve_atmosphere_32_fp64", "solve", 32, 32, 32, 4, "fp64", "atmosphere", max_iter=2000),
        # a spectrum: 16 bins of a stratified atmosphere (some bins nearly pure scattering), a fixed
        # number of iterations as a run over many snapshots affords
        c("spectrum_64x16_mixed", "solve", 64, 64, 64, 4, "mixed", "spectrum", nf=16, max_iter=60),
        # an odd-sized, bounded domain: rows that are no multiple of a vector, few planes
        c("solve_ragged_90x70x53_mixed", "solve", 90, 70, 53, 6, "mixed", "atmosphere", eps=0.1, max_iter=40),
        # the 128^3 turbulent box with 80 rays to convergence, mixed: the typical production solve
        c("solve_box_128_mixed", "solve", 128, 128, 128, 8, "mixed", "box", max_iter=1000),
        # the same structure on the plain FP64 path
        c("solve_box_96_fp64", "solve", 96, 96, 96, 6, "fp64", "box", tol=1e-4, max_iter=200),
        # a 2D plane with 4 bins
        c("plane_512x512x4_mixed", "solve", 512, 512, 1, 6, "mixed", "plane", nf=4, eps=0.05, max_iter=100),
        # second-order interpolation (sharp beams, shadows)
        c("quadratic_96_mixed", "solve", 96, 96, 96, 6, "mixed", "box", max_iter=12, interp="quadratic"),
        # requests of different sizes batched into shared launches
        c("many_8_mixed", "many", 64, 64, 64, 6, "mixed", "box", max_iter=400),
        # the largest: 256^3, 48 rays, eps = 1e-3; as many iterations as a pass may take
        c("large_256_mixed", "solve", 256, 256, 256, 6, "mixed", "turbulent_atmosphere", eps=1e-3, max_iter=40),
    ]


#: cell * ray * bin * formal solution of a drawn case, at most (the largest listed case has 3.2e10)
DRAW_MOST = 2.5e10


def draw(rng):
    def size(lo, hi, even=0.5):
        n = int(round(math.exp(rng.uniform(math.log(lo), math.log(hi)))))
        return max(lo, n // 4 * 4) if rng.random() < even else n

    while True:
        kind = rng.choice(["noalloc", "formal", "medium", "step", "solve", "solve", "solve", "many"])
        prec = rng.choice(["mixed", "mixed", "mixed", "fp64"])
        medium = rng.choice(["atmosphere", "box", "turbulent_atmosphere", "spectrum", "plane"])
        n_mu = rng.choice([4, 6, 8])
        nf = rng.choice([1, 1, 4, 16])
        top = {"noalloc": 48, "many": 96}.get(kind, 160 if prec == "mixed" else 96)
        if medium == "plane" and kind != "many":
            nx, ny, nz = size(64, 700), size(64, 700), 1
        else:
            medium = rng.choice(["atmosphere", "box"]) if medium == "plane" else medium
            nx, ny, nz = size(16, top), size(16, top), size(16, top)
            if rng.random() < 0.5:
                ny = nx
        interp = rng.choice(["linear", "linear", "linear", "quadratic"]) if kind in ("formal", "solve") else "linear"
        its = {"step": rng.randint(1, 8), "solve": int(round(math.exp(rng.uniform(math.log(10), math.log(300))))),
               "many": 100}.get(kind, 1)
        c = _case(kind, nx, ny, nz, n_mu, prec, medium, nf=nf, eps=round(10 ** rng.uniform(-3, -0.5), 6),
                  tol=10.0 ** -rng.randint(4, 7), max_iter=its, interp=interp)
        w = _updates(c) * (_iterations(c) + 1) * (12 if prec == "fp64" or interp == "quadratic" else 2)
        # (the call without allocations takes problems of at most 64 MB of working memory)
        if w <= DRAW_MOST and _updates(c) <= 1e9 and (kind != "noalloc" or _cells(c) * nf <= 24000):
            return c


# ---------------------------------------------------------------- sizes of the work

def _cells(c):
    return c["nx"] * c["ny"] * c["nz"]


def _rays(c):
    return c["n_mu"] * (c["n_mu"] + 2) // (2 if c["nz"] == 1 else 1)


def _members(c):
    """The problems of a ``many`` case: the case's size and smaller ones, odd ones among them."""
    if c["kind"] != "many":
        return [c]
    out = []
    for k, s in enumerate((1.0, 0.8, 0.5, 0.77, 0.5, 0.66, 0.9, 0.4)):
        n = [max(8, int(c[a] * s)) for a in ("nx", "ny", "nz")]
        out.append(dict(c, kind="solve", nx=n[0], ny=n[1], nz=n[2], n_mu=(c["n_mu"], 4)[k % 2]))
    return out


def _updates(c):
    return sum(m["nf"] * _cells(m) * _rays(m) for m in _members(c))


def _iterations(c):
    """Formal solutions of a pass (for converging solves, about as many as they take)."""
    if c["kind"] in ("noalloc", "formal", "medium"):
        return 1
    typical = 130 if c["medium"] == "box" else int(20 / math.sqrt(c["eps"]))
    return min(c["max_iter"], typical) if c["tol"] <= 1e-6 else min(c["max_iter"], typical * 2 // 3)


def work(c):
    n = sum(m["nf"] * _cells(m) for m in _members(c))
    outs = {"noalloc": 1, "formal": 2, "medium": 1, "step": 5, "solve": 17, "many": 2}[c["kind"]]
    ins = {"noalloc": 3, "formal": 1, "medium": 4, "step": 4, "solve": 3, "many": 0}[c["kind"]]
    # per update: the interpolants of S and I on the upwind face (14), the segment (5), the angle sum
    # (2); once per medium the interpolant of chi, the optical depth and the two weights (13)
    flops = _updates(c) * (21.0 * _iterations(c) + 13.0)
    if c["interp"] == "quadratic":   # five 3 x 3 interpolants, the control value, its weights
        flops = _updates(c) * 200.0 * _iterations(c)
    return {"bytes": 8.0 * n * (ins + outs), "flops": flops}


# ------------------------------------------------------------------------- inputs

def _field(shape, gen, slope=-11.0 / 3.0):
    """Unit-variance periodic Gaussian random field with power spectrum k^slope, [z][y][x]."""
    white = torch.randn(shape, generator=gen, dtype=F64, device=DEV)
    k = [torch.fft.fftfreq(n, d=1.0 / n, dtype=F64, device=DEV) for n in shape[:2]]
    kx = torch.fft.rfftfreq(shape[2], d=1.0 / shape[2], dtype=F64, device=DEV)
    k2 = k[0][:, None, None] ** 2 + k[1][None, :, None] ** 2 + kx[None, None, :] ** 2
    amp = torch.where(k2 > 0, k2.clamp(min=1e-30) ** (slope / 4.0), torch.zeros_like(k2))
    g = torch.fft.irfftn(torch.fft.rfftn(white) * amp, s=shape, dim=(0, 1, 2))
    g = g - g.mean()
    return g / g.std()


def _profile(n, tau_top=1e-4, tau_bot=1e3):
    """Exponential atmosphere: optical depth log-spaced from the bottom (first) to the top, chi per cell."""
    r = (tau_bot / tau_top) ** (1.0 / (n - 1))
    tau = tau_top * r ** torch.arange(n - 1, -1, -1, dtype=F64, device=DEV)
    return tau * math.log(r)


def _faces(c):
    if c["medium"] == "box":
        return (P, P, P), (P, P, P)
    if c["medium"] == "plane":
        return (P, T, P), (P, V, P)
    return (P, P, T), (P, P, V)


def _medium(c, gen):
    """chi, eps, B [nf][nz][ny][nx] and the frequency weights."""
    nx, ny, nz, nf = c["nx"], c["ny"], c["nz"], c["nf"]
    g = _field((nz, ny, nx), gen)
    h = _field((nz, ny, nx), gen)
    scale = (1.0 + torch.arange(nf, dtype=F64, device=DEV) / nf)[:, None, None, None]
    weights = torch.full((nf,), 1.0 / nf, dtype=F64, device=DEV)
    if c["medium"] == "box":                    # log-normal density and temperature, box depth about 30
        rho, tem = torch.exp(g - 0.5), torch.exp(0.3 * h - 0.045)
        chi_a, chi_s = 0.1 * rho ** 2 * tem ** -3.5, 0.9 * rho
        chi = chi_a + chi_s
        eps = (chi_a / chi).expand(nf, -1, -1, -1)
        chi = (chi * (30.0 / (chi.mean() * max(nx, ny, nz)))) * scale
        B = tem ** 4 / scale
    elif c["medium"] == "spectrum":             # free-free absorption over log-spaced bins, grey scattering
        sc = _profile(nz)[:, None, None] * torch.exp(0.1 * g)
        tem = torch.exp(0.1 * h)
        x = torch.exp(torch.linspace(math.log(0.01), math.log(30.0), nf, dtype=F64, device=DEV)) if nf > 1 \
            else torch.ones(1, dtype=F64, device=DEV)
        x = x[:, None, None, None]
        chi_a = 1e-2 * sc ** 2 / sc.max() * tem ** -0.5 * x ** -3 * -torch.expm1(-x / tem)
        chi = chi_a + sc
        eps = chi_a / chi
        B = x ** 3 / torch.expm1(x / tem)
        if nf > 1:
            d = torch.diff(x.flatten())
            weights = 0.5 * (torch.cat([d, d[-1:] * 0]) + torch.cat([d[:1] * 0, d]))
    else:
        if c["medium"] == "plane":              # stratified along y
            prof, amp = _profile(ny)[None, :, None], 0.1
        else:
            prof = _profile(nz)[:, None, None]
            amp = 1.0 if c["medium"] == "turbulent_atmosphere" else 0.1
        tem = torch.exp(0.3 * amp * h - 0.045 * amp * amp)
        chi = prof * torch.exp(amp * g - 0.5 * amp * amp) * scale
        eps = torch.full_like(chi, c["eps"])
        B = tem ** 4 / scale
    full = (nf, nz, ny, nx)
    return [a.expand(full).contiguous() for a in (chi, eps, B)] + [weights]


def _generator(seed):
    gen = torch.Generator(device=DEV)
    gen.manual_seed(int(seed) * 7919 + 17)
    return gen


def _inputs(c, seed):
    """Per member problem (chi, eps, B, weights, S): S a source function as an outer iteration has it."""
    gen, out = _generator(seed), []
    for m in _members(c):
        chi, eps, B, w = _medium(m, gen)
        S = B * (0.6 + 0.4 * torch.rand(B.shape, generator=gen, dtype=F64, device=DEV))
        out.append((chi, eps, B, w, S))
    return out


def prepare(c, seed):
    state = {"case": c, "inputs": _inputs(c, seed), "grids": []}
    if c["kind"] == "noalloc":
        chi = state["inputs"][0][0]
        state["J"] = torch.empty_like(chi)
        return state
    for m, (chi, eps, B, w, S) in zip(_members(c), state["inputs"]):
        lo, hi = _faces(m)
        g = rt.Grid(m["nx"], m["ny"], m["nz"], n_mu=m["n_mu"], nfreq=m["nf"], bc_lo=lo, bc_hi=hi, prec=m["prec"])
        if m["interp"] != "linear":
            g.set_interpolation(m["interp"])
        if c["kind"] in ("formal", "many"):     # a medium that stands
            g.set_opacity_source(chi, eps, B, w)
        state["grids"].append(g)
    return state


# -------------------------------------------------------------------------- a pass

def _kept(c, *arrays):
    return [a.float() if c["prec"] == "mixed" else a for a in arrays]


def run(state):
    c = state["case"]
    chi, eps, B, w, S = state["inputs"][0]
    if c["kind"] == "noalloc":
        lo, hi = _faces(c)
        J = rt.formal_solve_noalloc(c["nx"], c["ny"], c["nz"], chi, S, B, state["J"], n_mu=c["n_mu"],
                                    nfreq=c["nf"], bc_lo=lo, bc_hi=hi, prec=c["prec"])
        return {"J": _kept(c, J)[0]}
    g = state["grids"][0]
    if c["kind"] == "formal":
        J, L = g.formal_solve(S, want_lstar=True)
        return dict(zip(("J", "lstar"), _kept(c, J, L)))
    if c["kind"] == "medium":
        g.set_opacity_source(chi, eps, B, w)
        return {"J": _kept(c, g.formal_solve(S))[0]}
    if c["kind"] == "many":
        res = rt.ali_solve_many(state["grids"], tol=c["tol"], max_iter=c["max_iter"], raise_on_fail=False)
        return {"S": [_kept(c, x.get_S(on_device=True))[0] for x in state["grids"]], "iters": [r[0] for r in res]}
    # the steps and solves: the new medium, the iteration, the outputs
    g.set_opacity_source(chi, eps, B, w)
    step = c["kind"] == "step"
    iters, _, _ = g.ali_solve(S if step else None, tol=c["tol"], max_iter=c["max_iter"], raise_on_fail=False)
    m = g.moments(on_device=True, want=("J", "H", "Q") if step else ("J", "H", "K", "f", "Q"))
    out = dict(zip(m, _kept(c, *m.values())))
    out["S"] = _kept(c, g.get_S(on_device=True))[0]
    out["iters"] = iters
    return out


# ------------------------------------------------- the same in plain torch, 64 bits
# The equations as include/rt_sc.h states them (Davis, Stone & Jiang 2012: the
# update Eq. 20, the moments Eqs. 17-19, the Jacobi iteration Eqs. 24-25), plane by
# plane over all rays that cross the same face.

def _angles(n_mu, two_d):
    """Level-symmetric set: mu_i^2 = a + (i-1) 2 (1-3a)/(n-2), one weight per permutation class, from
    sum w = 1 and the even moments 1/(2p+1), by Newton's method from the tabulated values."""
    half = n_mu // 2
    nodes = [(i, j, half + 2 - i - j) for i in range(1, half + 1) for j in range(1, half + 1) if half + 2 - i - j >= 1]
    classes = sorted({tuple(sorted(n)) for n in nodes})
    cls = np.array([classes.index(tuple(sorted(n))) for n in nodes])
    lev = np.array([n[2] - 1 for n in nodes])
    mu1, wc = {4: (0.3500212, [1.0 / 3.0]), 6: (0.2666355, [0.1761263, 0.1572071]),
               8: (0.2182179, [0.1209877, 0.0907407, 0.0925926])}[n_mu]
    nc = len(classes)

    def residual(x):
        mu2 = x[0] + lev * 2.0 * (1.0 - 3.0 * x[0]) / (n_mu - 2)
        wn = x[1:][cls]
        return np.array([wn.sum() - 1.0] + [(wn * mu2 ** p).sum() - 1.0 / (2 * p + 1) for p in range(2, nc + 2)])

    x = np.array([mu1 ** 2] + wc)
    for _ in range(8):
        jac = np.stack([residual(x + 1e-30j * e).imag / 1e-30 for e in np.eye(nc + 1)], axis=1)
        x = x - np.linalg.solve(jac, residual(x))
    level = np.sqrt(x[0] + np.arange(half) * 2.0 * (1.0 - 3.0 * x[0]) / (n_mu - 2))
    mu, wq = [], []
    for o in range(4 if two_d else 8):
        sign = np.array([-1.0 if o & 1 else 1.0, -1.0 if o & 2 else 1.0, -1.0 if o & 4 else 1.0])
        for n, k in zip(nodes, cls):
            mu.append(sign * level[np.array(n) - 1])
            wq.append(x[1 + k] / 8.0 * (2.0 if two_d else 1.0))
    return np.array(mu), np.array(wq)


_ROLES = {0: (1, 2), 1: (0, 2), 2: (0, 1)}          # sweep axis -> plane axes (u, v)


def _to_planes(a, axis):
    """[..., z, y, x] -> [..., w, v, u]."""
    return a if axis == 2 else (a.transpose(-3, -2) if axis == 1 else a.permute(*range(a.dim() - 3), -1, -3, -2))


def _from_planes(a, axis):
    return a if axis == 2 else (a.transpose(-3, -2) if axis == 1 else a.permute(*range(a.dim() - 3), -2, -1, -3))


class _Exact:
    """Formal solutions and the Jacobi iteration.  The rays that cross the face of one axis go together, each
    in coordinates flipped so that it runs towards larger indices: [bin][ray][w][v][u]."""

    def __init__(self, c, chi, eps, B, w):
        self.c, self.chi, self.eps, self.B, self.fw = c, chi, eps, B, w
        self.two_d = c["nz"] == 1
        self.n = (c["nx"], c["ny"], c["nz"])
        lo, hi = _faces(c)
        self.bc = list(zip(lo, hi))
        if self.two_d:
            self.bc[2] = (P, P)
        self.mu, self.wq = _angles(c["n_mu"], self.two_d)
        path = 1.0 / np.abs(self.mu)
        if self.two_d:
            path[:, 2] = np.inf
        axis = np.argmin(path, axis=1)
        self.sets = []
        for a in range(3):
            k = np.flatnonzero(axis == a)
            if len(k):
                s = path[k, a]
                f = [np.minimum(1.0, s * np.abs(self.mu[k, b])) if np.isfinite(path[k, b]).all() else 0.0 * s
                     for b in _ROLES[a]]
                self.sets.append((a, k, *(torch.from_numpy(x).to(DEV)[None, :, None, None, None] for x in (s, *f))))
        self.I, self.weights = {}, {}

    def _flips(self, a, k):
        u, v = _ROLES[a]
        return [d for d, b in ((-3, a), (-2, v), (-1, u)) if self.mu[k, b] < 0]

    def _per_ray(self, x, a, ks):
        x = _to_planes(x, a)
        return torch.stack([torch.flip(x, self._flips(a, k)) for k in ks], dim=1)

    def _index(self, a):
        n = self.n[a]
        ends = (n - 1, 0) if self.bc[a][0] == P else (0, n - 1)
        return torch.tensor([ends[0], *range(n), ends[1]], device=DEV)

    def _padded(self, x, a):
        for d, b in ((-3, a), (-2, _ROLES[a][1]), (-1, _ROLES[a][0])):
            x = x.index_select(d, self._index(b))
        return x

    def _thermal(self, b, ks, downwind):
        """Per ray: 1 where the face of axis b that it comes from (goes to) is thermal, 0 where vacuum."""
        side = [self.bc[b][int((self.mu[k, b] < 0) != downwind)] for k in ks]
        return torch.tensor([1.0 if x == T else 0.0 for x in side], dtype=F64, device=DEV)[None, :, None]

    def _at(self, x, a, dw, dv, du):
        nw, nv, nu = self.n[a], self.n[_ROLES[a][1]], self.n[_ROLES[a][0]]
        return x[..., 1 + dw:1 + dw + nw, 1 + dv:1 + dv + nv, 1 + du:1 + du + nu]

    def _segments(self, S, a, ks, s, fu, fv):
        """Attenuation, the source's contribution and the weight of S at the cell, for every ray and cell."""
        if self.c["interp"] == "quadratic":
            return self._quadratic(S, a, ks, s, fu, fv)

        def face(x):
            x = self._padded(x, a)
            return (1 - fv) * ((1 - fu) * self._at(x, a, -1, 0, 0) + fu * self._at(x, a, -1, 0, -1)) + \
                fv * ((1 - fu) * self._at(x, a, -1, -1, 0) + fu * self._at(x, a, -1, -1, -1))

        if a not in self.weights:
            chi = self._per_ray(self.chi, a, ks)
            tau = (face(chi) + chi) * (s / 2)
            small = tau * (1 / 2 - tau * (1 / 6 - tau * (1 / 24 - tau * (1 / 120 - tau * (1 / 720 - tau * (1 / 5040))))))
            psi = torch.where(tau < 1e-2, small, 1 + torch.expm1(-tau) / tau.clamp(min=1e-9))
            self.weights[a] = (torch.exp(-tau), psi)
        E, psi = self.weights[a]
        S0 = self._per_ray(S, a, ks)
        Sm = face(S0)
        return E, Sm - E * Sm + psi * (S0 - Sm), psi

    def _quadratic(self, S, a, ks, s, fu, fv):
        chi, S0 = self._per_ray(self.chi, a, ks), self._per_ray(S, a, ks)

        def face(x, dw, tu, tv):
            x = self._padded(x, a)
            rows = [_parabola(*(self._at(x, a, dw, r, q) for q in (-1, 0, 1)), tu) for r in (-1, 0, 1)]
            return _parabola(*rows, tv)

        Sm, Sp = face(S0, -1, -fu, -fv), face(S0, 1, fu, fv)
        hm, hp = (face(chi, -1, -fu, -fv) + chi) * (s / 2), (chi + face(chi, 1, fu, fv)) * (s / 2)
        Sc = S0 - 0.5 * hm * (hp * ((S0 - Sm) / hm) + hm * ((Sp - S0) / hp)) / (hm + hp)
        dSc = (1 - 0.5 * hm * (hp / hm - hm / hp) / (hm + hp)).clamp(0, 1)
        lo, hi = torch.minimum(Sm, S0), torch.maximum(Sm, S0)
        below, above = Sc < lo, Sc > hi
        dSc = torch.where(below, (lo == S0).to(F64), torch.where(above, (hi == S0).to(F64), dSc))
        Sc = torch.minimum(torch.maximum(Sc, lo), hi)
        # m_n = int_0^t x^n e^-x dx / t^(n+1)
        E = torch.exp(-hm)
        E0 = -torch.expm1(-hm)
        E1 = E0 - hm * E
        small, x, m = hm < 0.5, hm.clamp(max=0.5), []
        for n, direct in enumerate((E0 / hm, E1 / hm ** 2, (2 * E1 - hm * hm * E) / hm ** 3)):
            p, total = torch.ones_like(x), torch.zeros_like(x)
            for q in range(16):
                total = total + p / (math.factorial(q) * (q + n + 1))
                p = p * -x
            m.append(torch.where(small, total, direct))
        b, g = hm * (m[0] - 2 * m[1] + m[2]), 2 * hm * (m[1] - m[2])
        return E, hm * m[2] * Sm + b * S0 + g * Sc, b + g * dSc

    def formal(self, S):
        """One formal solution from the intensities of the last one (first: the image cells' S): J, Lambda*."""
        J, lam = torch.zeros_like(S), torch.zeros_like(S)
        quadratic = self.c["interp"] == "quadratic"
        for a, ks, s, fu, fv in self.sets:
            u, v = _ROLES[a]
            nw, nv, nu = self.n[a], self.n[v], self.n[u]
            iu, iv = self._index(u), self._index(v)
            E, src, psi = self._segments(S, a, ks, s, fu, fv)
            old = self.I.get(a)
            if old is None:
                old = self._per_ray(S, a, ks)
            faces = [(b, self._thermal(b, ks, False), self._thermal(b, ks, True)) for b in range(3) if self.bc[b][0] != P]
            Bp = self._per_ray(self.B, a, ks).index_select(-1, iu).index_select(-2, iv) if faces else None
            new = torch.empty_like(E)
            gu, gv = fu[..., 0], fv[..., 0]
            for w in range(nw):
                wm = w - 1 if w else (nw - 1 if self.bc[a][0] == P else 0)
                lag = old[:, :, wm]
                I = lag.index_select(-1, iu).index_select(-2, iv)
                # a periodic face keeps one intensity per cell and ray, its outflow: the second-order stencil's
                # ghosts on the downstream side read it too (the first out-of-range axis in the order z, y, x)
                if self.bc[v][0] == P and (w or a != 2):
                    I[..., 0, :] = I[..., -1, :] = lag[..., nv - 1, :].index_select(-1, iu)
                if self.bc[u][0] == P and (w or a == 0):
                    I[..., 1:-1, 0] = I[..., 1:-1, -1] = lag[..., nu - 1]
                if w:
                    I[..., 1:-1, 1:-1] = new[:, :, w - 1]
                for b, up, down in faces:        # past several bounded faces z decides, then y, then x
                    if b == a and w == 0:
                        I = Bp[:, :, wm] * up[..., None]
                    elif b == u:
                        I[..., 0], I[..., -1] = Bp[:, :, wm, :, 0] * up, Bp[:, :, wm, :, -1] * down
                    elif b == v:
                        I[..., 0, :], I[..., -1, :] = Bp[:, :, wm, 0] * up, Bp[:, :, wm, -1] * down
                if quadratic:
                    rows = [_parabola(*(I[..., r:r + nv, q:q + nu] for q in range(3)), -gu) for r in range(3)]
                    Im = _parabola(*rows, -gv)
                else:
                    row = (1 - gu) * I[..., :nv + 1, 1:1 + nu] + gu * I[..., :nv + 1, :nu]
                    Im = (1 - gv) * row[..., 1:, :] + gv * row[..., :-1, :]
                new[:, :, w] = E[:, :, w] * Im + src[:, :, w]
            self.I[a] = new
            for i, k in enumerate(ks):
                J += self.wq[k] * _from_planes(torch.flip(new[:, i], self._flips(a, k)), a)
                lam += self.wq[k] * _from_planes(torch.flip(psi[:, i], self._flips(a, k)), a)
        return J, lam

    def moments(self):
        """H [bin][3], K [bin][6] (xx, yy, zz, xy, xz, yz) of the last formal solution."""
        out = torch.zeros((self.chi.shape[0], 9) + self.chi.shape[1:], dtype=F64, device=DEV)
        for a, ks, *_ in self.sets:
            for i, k in enumerate(ks):
                x, y, z = self.mu[k]
                I = self.wq[k] * _from_planes(torch.flip(self.I[a][:, i], self._flips(a, k)), a)
                for q, r in enumerate((x, y, z, x * x, y * y, z * z, x * y, x * z, y * z)):
                    out[:, q] += r * I
        if self.two_d:
            out[:, [2, 7, 8]] = 0.0
        return out[:, :3], out[:, 3:]

    def solve(self, S, tol, max_iter):
        for it in range(1, max_iter + 1):
            J, lam = self.formal(S)
            dS = ((1 - self.eps) * J + self.eps * self.B - S) / (1 - (1 - self.eps) * lam)
            S = S + dS
            if float((dS.abs() / S.abs()).max()) <= tol:
                break
        return S, J, it


def _parabola(fm, f0, fp, t):
    """Through three values at t in [-1, 1], clamped to the two that bracket t."""
    val = f0 + 0.5 * t * (fp - fm) + 0.5 * t * t * (fp - 2 * f0 + fm)
    fe = torch.where(t < 0, fm, fp)
    val = torch.minimum(torch.maximum(val, torch.minimum(fe, f0)), torch.maximum(fe, f0))
    return torch.where(t == 0, f0, val)


def exact(c, seed):
    members = _members(c)
    # (about 15 small launches a plane, and the traffic of their temporaries)
    seconds = sum((_iterations(m) + 1) * (3e-4 * (m["nx"] + m["ny"] + m["nz"]) + 2.5e-10 * _updates(m)) *
                  (4 if m["interp"] == "quadratic" else 1) for m in members)
    if seconds > 20:
        return None
    inputs = _inputs(c, seed)
    if c["kind"] == "many":
        got = [_Exact(m, *x[:4]).solve(x[2], m["tol"], m["max_iter"]) for m, x in zip(members, inputs)]
        return {"S": [r[0] for r in got], "iters": [r[2] for r in got]}
    chi, eps, B, w, S = inputs[0]
    E = _Exact(c, chi, eps, B, w)
    if c["kind"] in ("noalloc", "formal", "medium"):
        J, lam = E.formal(S)
        return {"J": J, "lstar": lam} if c["kind"] == "formal" else {"J": J}
    S, J, iters = E.solve(S if c["kind"] == "step" else B, c["tol"], c["max_iter"])
    H, K = E.moments()
    got = {"J": J, "H": H, "S": S, "iters": iters,
           "Q": 4 * math.pi * (w[:, None, None, None] * eps * chi * (J - B)).sum(0)}
    if c["kind"] == "solve":
        got.update(K=K, f=K / J[:, None])
    return got
