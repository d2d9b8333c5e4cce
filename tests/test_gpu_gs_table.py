"""The reverse phase of FP64 Gauss-Seidel reads the streamed sweep's weight table (row
segments of two cells: rows of 1, 2, 3 and 10 cells): the first iterations against the
oracle's, as in test_gpu_gauss_seidel (1e-11)."""
import numpy as np
import pytest

from oracle import oracle as O
from paper_1201_2222_gb300 import workloads as W

torch = pytest.importorskip("torch")
pytestmark = pytest.mark.gpu

P, V, T = 0, 1, 2


@pytest.mark.parametrize("nx,ny,nz,nf", [(1, 4, 5, 2), (2, 3, 4, 1), (3, 5, 4, 2), (10, 7, 6, 2), (9, 6, 1, 2)])
def test_first_iterations(nx, ny, nz, nf):
    from paper_1201_2222_gb300 import build, rt
    if not torch.cuda.is_available():
        pytest.skip("no CUDA device")
    build.build()
    lo, hi = ((P, P, T), (P, P, V)) if nz > 1 else ((P, T, P), (P, V, P))
    p = W.random_box(nx, ny, nz, seed=500 + nx, n_mu=4, nf=nf, bc_lo=lo, bc_hi=hi)
    og = O.Grid.from_problem(p)
    with rt.Grid.from_problem(p, prec="fp64") as g:
        g.set_iteration("gauss_seidel")
        g.set_opacity_source(p.chi, p.eps, p.B, p.freq_w)
        for n in (1, 3):
            g.ali_solve(tol=0.0, max_iter=n, raise_on_fail=False)
            ref = O.ali_solve(og, p.chi, p.eps, p.B, p.freq_w, tol=0.0, max_iter=n, moments=False,
                              method="gauss_seidel")
            assert np.max(np.abs(g.get_S() / ref["S"] - 1)) < 1e-11
        assert g.sweep_table()["streams"]
