"""An error of the CUDA runtime that a call has returned is not returned again by the
next call, on another grid."""
import numpy as np
import pytest

from oracle import oracle as O
from paper_1201_2222_gb300 import workloads as W

torch = pytest.importorskip("torch")
pytestmark = pytest.mark.gpu


def test_out_of_memory_is_reported_once():
    from paper_1201_2222_gb300 import build, rt
    if not torch.cuda.is_available():
        pytest.skip("no CUDA device")
    build.build()
    p = W.random_box(6, 5, 4, seed=700, n_mu=2)
    with rt.Grid.from_problem(p, prec="fp64") as g:
        with pytest.raises(rt.RTError) as e:
            rt.Grid(4096, 4096, 4096, n_mu=2)            # 550 GB a field
        assert e.value.status == rt.RT_ERR_OOM
        g.set_opacity_source(p.chi, p.eps, p.B, p.freq_w)
        J = g.formal_solve(p.B)
    ref = O.formal_solution(O.Grid.from_problem(p), p.chi[0], p.B[0], p.B[0])["J"]
    assert np.max(np.abs(J[0] / ref - 1)) < 1e-10
