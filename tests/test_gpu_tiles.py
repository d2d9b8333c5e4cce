"""The kernels that work on tiles of cells -- Lambda*, the Jacobi update, the
reduction of moment partials, the smallest epsilon of the thick cells -- at the edges
of their tiles, and the FP64 segment weights on both sides of their branch."""
import numpy as np
import pytest

from oracle import oracle as O
from paper_1201_2222_gb300 import workloads as W

torch = pytest.importorskip("torch")
pytestmark = pytest.mark.gpu

P, V, T = 0, 1, 2

CASES = [   # nx, ny, nz, n_mu, bc_lo, bc_hi: below, at and beyond 32 x 16 and 32 x 32; few and many tiles
    (1, 1, 3, 4, (P, P, T), (P, P, V)),
    (31, 15, 2, 4, (P, T, P), (P, V, P)),
    (32, 16, 3, 6, (V, P, T), (T, P, V)),
    (33, 33, 4, 4, (P, P, P), (P, P, P)),
    (36, 34, 90, 2, (P, P, T), (P, P, V)),
    (64, 8, 160, 2, (P, P, T), (P, P, V)),
]


@pytest.fixture(scope="module")
def rt():
    if not torch.cuda.is_available():
        pytest.skip("no CUDA device")
    from paper_1201_2222_gb300 import build, rt as _rt
    build.build()
    return _rt


def rel(a, b):
    a, b = np.asarray(a), np.asarray(b)
    return float(np.max(np.abs(a - b) / np.maximum(np.abs(b), 1e-300)))


@pytest.mark.parametrize("prec", ["fp64", "mixed"])
@pytest.mark.parametrize("case", range(len(CASES)))
def test_lambda_star_updates_and_moments(rt, prec, case):
    """Rounding only: 1e-10 FP64, 1e-5 float32; the moments are sums of positive terms
    (J, f's diagonal) or bounded by J (H)."""
    nx, ny, nz, n_mu, lo, hi = CASES[case]
    nf = 2 if case % 2 else 1
    p = W.random_box(nx, ny, nz, seed=700 + case, n_mu=n_mu, nf=nf, bc_lo=lo, bc_hi=hi)
    og = O.Grid.from_problem(p)
    tol = 1e-10 if prec == "fp64" else 1e-5
    with rt.Grid.from_problem(p, prec=prec) as g:
        g.set_sweep_config(variant=3)
        g.set_opacity_source(p.chi, p.eps, p.B, p.freq_w)
        _, L = g.formal_solve(p.B, want_lstar=True)
        for f in range(nf):
            assert rel(L[f], O.formal_solution(og, p.chi[f], p.B[f], p.B[f])["lstar"]) < tol
        it, _, _ = g.ali_solve(tol=1e-7, max_iter=12, raise_on_fail=False)
        ref = O.ali_solve(og, p.chi, p.eps, p.B, p.freq_w, tol=1e-7, max_iter=12)
        m = g.moments()
        assert it == ref["iters"]
        assert rel(g.get_S(), ref["S"]) < tol
        assert rel(m["J"], ref["J"]) < tol
        assert rel(m["K"][:, :3], ref["K"][:, :3]) < tol
        assert np.max(np.abs(m["H"] - ref["H"]) / ref["J"][:, None]) < tol


@pytest.mark.parametrize("tau", [1e-4, 0.0099, 0.0101, 0.3, 0.499, 0.501, 0.9, 7.0, 60.0])
def test_fp64_weights_at_their_branches(rt, tau):
    """Lambda* of a uniform periodic medium is sum_k w_k Psi0(chi s_k).  Psi0 is good to
    1e-15, chi s to another 1e-15 (interpolation, path length), and the sum of na
    positive terms adds na rounding errors of 1.2e-16 at most."""
    n = 4
    z = np.full((1, n, n, n), tau)
    p = W.Problem(name="uniform", nx=n, ny=n, nz=n, n_mu=4, chi=z, eps=np.full_like(z, 0.5), B=np.ones_like(z),
                  freq_w=np.ones(1), bc_lo=(P, P, P), bc_hi=(P, P, P))
    og = O.Grid.from_problem(p)
    with rt.Grid.from_problem(p, prec="fp64") as g:
        g.set_opacity_source(p.chi, p.eps, p.B, p.freq_w)
        _, L = g.formal_solve(p.B, want_lstar=True)
    x = np.longdouble(tau) * (1 / np.max(np.abs(og.mu), axis=1)).astype(np.longdouble)
    want = float(np.sum(np.asarray(og.w, dtype=np.longdouble) * (1 + np.expm1(-x) / x)))
    # (1 + expm1(-x)/x in the 64-bit mantissa of x86 loses 1e-19/x: 1e-14 at the thinnest)
    assert rel(L, want) < 2e-15 + og.na * 1.2e-16 + 1e-18 / tau
