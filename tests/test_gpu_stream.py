"""The streamed sweep (weights read from a table; variant 3, and FP64's automatic
choice) at the sizes where its work split can go wrong, against the oracle: rows of
one cell, shorter and longer than a warp's segments and of every remainder; strips
of one row, as many strips as a cluster holds; one, two and many planes; threads
with no segment and with several; every kind of face.  Tolerances as in
test_gpu_parity (rounding only: 1e-10 FP64, 1e-5 float32)."""
import numpy as np
import pytest

from oracle import oracle as O
from paper_1201_2222_gb300 import workloads as W

torch = pytest.importorskip("torch")
pytestmark = pytest.mark.gpu

P, V, T, F = 0, 1, 2, 3

CASES = [
    # (nx, ny, nz, n_mu, bc_lo, bc_hi, sweep config)
    (1, 1, 2, 4, (P, P, T), (P, P, V), {}),
    (1, 7, 3, 2, (V, P, T), (T, P, V), dict(cluster_ctas=3)),
    (2, 2, 2, 6, (P, P, P), (P, P, P), dict(angles_per_group=8, cluster_ctas=2)),
    (133, 5, 4, 4, (P, P, T), (P, P, V), dict(cluster_ctas=4)),
    (132, 8, 5, 4, (P, T, P), (P, V, P), dict(angles_per_group=1, cluster_ctas=5)),
    (40, 36, 17, 6, (P, P, P), (P, P, P), dict(angles_per_group=3, cluster_ctas=16)),
    (36, 40, 33, 8, (T, V, P), (V, T, P), dict(angles_per_group=7, cluster_ctas=2, threads=64)),
    (30, 31, 29, 4, (T, T, V), (T, V, T), dict(angles_per_group=2, cluster_ctas=1, threads=32)),
    (260, 67, 1, 6, (P, T, P), (P, V, P), dict(angles_per_group=2)),
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
def test_formal_solutions_and_iterations(rt, prec, case):
    nx, ny, nz, n_mu, lo, hi, cfg = CASES[case]
    p = W.random_box(nx, ny, nz, seed=300 + case, n_mu=n_mu, nf=2 if case % 2 else 1, bc_lo=lo, bc_hi=hi)
    og = O.Grid.from_problem(p)
    tol = 1e-10 if prec == "fp64" else 1e-5
    with rt.Grid.from_problem(p, prec=prec) as g:
        if cfg:
            g.set_sweep_config(**cfg)
        g.set_opacity_source(p.chi, p.eps, p.B, p.freq_w)
        S = np.random.default_rng(case).uniform(0.3, 2.0, p.chi.shape)
        G = [O.init_ghosts(og, S[f]) for f in range(p.nf)]
        for k in range(3):                       # the later ones from lagged periodic ghosts
            J = g.formal_solve(S if k == 0 else None)
            for f in range(p.nf):
                ref = O.formal_solution(og, p.chi[f], S[f], p.B[f], G_prev=G[f])
                G[f] = ref["G_next"]
                assert rel(J[f], ref["J"]) < tol
        # increments (float32), the ghosts they advance, and the moments
        it, _, _ = g.ali_solve(tol=1e-6, max_iter=60, raise_on_fail=False)
        ref = O.ali_solve(og, p.chi, p.eps, p.B, p.freq_w, tol=1e-6, max_iter=60)
        m = g.moments()
        assert it == ref["iters"]
        assert rel(g.get_S(), ref["S"]) < tol
        assert rel(m["J"], ref["J"]) < tol
        assert rel(m["K"][:, :3], ref["K"][:, :3]) < tol


@pytest.mark.parametrize("prec", ["fp64", "mixed"])
def test_fixed_faces_and_strips(rt, prec):
    """Incident intensities on a bounded face, the plane cut into strips of one row."""
    rng = np.random.default_rng(4)
    p = W.random_box(9, 6, 8, seed=321, n_mu=4, bc_lo=(F, P, T), bc_hi=(V, P, V))
    og = O.Grid.from_problem(p)
    I = rng.uniform(0.0, 2.0, (1, og.na, 8, 6))
    faces = [np.zeros(og.na * og.face[f // 2]) for f in range(6)]
    faces[0] = I.reshape(-1)
    with rt.Grid.from_problem(p, prec=prec) as g:
        g.set_sweep_config(angles_per_group=2, cluster_ctas=6)
        g.set_opacity_source(p.chi, p.eps, p.B, p.freq_w)
        g.set_boundary_intensity(0, I)
        J = g.formal_solve(p.B)
    ref = O.formal_solution(og, p.chi[0], p.B[0], p.B[0], G_prev=O.init_ghosts(og, p.B[0]),
                            I_fixed=np.concatenate(faces))
    assert rel(J[0], ref["J"]) < (1e-10 if prec == "fp64" else 1e-5)
