"""More frequency bins than a launch grid's z extent holds (65535): a formal solution and
its moments, bins on both sides of the limit against the oracle (1e-10 FP64, 1e-5
float32)."""
import numpy as np
import pytest

from oracle import oracle as O
from paper_1201_2222_gb300 import workloads as W

torch = pytest.importorskip("torch")
pytestmark = pytest.mark.gpu

P, V, T = 0, 1, 2


@pytest.mark.parametrize("prec", ["fp64", "mixed"])
def test_formal_solution_and_moments(prec):
    from paper_1201_2222_gb300 import build, rt
    if not torch.cuda.is_available():
        pytest.skip("no CUDA device")
    build.build()
    nf = 65539
    q = W.random_box(2, 1, 2, seed=510, n_mu=2, nf=7, bc_lo=(P, P, T), bc_hi=(P, P, V))
    rep = lambda a: np.ascontiguousarray(a[np.arange(nf) % 7])
    og = O.Grid.from_problem(q)
    tol = 1e-10 if prec == "fp64" else 1e-5
    with rt.Grid(2, 1, 2, n_mu=2, nfreq=nf, bc_lo=q.bc_lo, bc_hi=q.bc_hi, dx=q.dx, dy=q.dy, dz=q.dz, prec=prec) as g:
        g.set_opacity_source(rep(q.chi), rep(q.eps), rep(q.B))
        J = g.formal_solve(rep(q.B))
        m = g.moments(want=("J", "K"))
    refs = [O.formal_solution(og, q.chi[f], q.B[f], q.B[f], moments=True) for f in range(7)]
    for f in list(range(7)) + list(range(65529, nf)):
        ref = refs[f % 7]
        assert np.max(np.abs(J[f] / ref["J"] - 1)) < tol
        assert np.max(np.abs(m["J"][f] / ref["J"] - 1)) < tol
        assert np.max(np.abs(m["K"][f, :3] / ref["K"][:3] - 1)) < tol
