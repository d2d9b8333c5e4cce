"""rt_grid_footprint bounds what a grid allocates (the server admits requests by it)."""
import numpy as np
import pytest

from paper_1201_2222_gb300 import workloads as W

torch = pytest.importorskip("torch")
pytestmark = pytest.mark.gpu

P, V, T, F, X = 0, 1, 2, 3, 4


@pytest.fixture(scope="module")
def rt():
    if not torch.cuda.is_available():
        pytest.skip("no CUDA device")
    from paper_1201_2222_gb300 import build, rt as _rt
    build.build()
    return _rt


@pytest.mark.parametrize("prec", ["fp64", "mixed"])
@pytest.mark.parametrize("table", [-1, 0])
@pytest.mark.parametrize("shape,n_mu", [((32, 32, 32), 8), ((30, 21, 17), 6), ((96, 96, 96), 8)])
def test_many_rays(rt, prec, table, shape, n_mu):
    """The arrays that grow with the groups, and the others of some size: J and nine
    moments a group, 13 (11) fields, the moments' outputs, the tables; of the FP64
    iterations' grid 17 fields."""
    p = W.random_box(*shape, seed=600, n_mu=n_mu, eps_range=(0.3, 1.0))
    N, na, ts = p.chi.size, n_mu * (n_mu + 2), 4 if prec == "mixed" else 8
    with rt.Grid.from_problem(p, prec=prec) as g:
        g.set_opacity_source(p.chi, p.eps, p.B, p.freq_w)
        g.set_table_limit(table)
        g.ali_solve(tol=1e-6, max_iter=2, raise_on_fail=False)
        g.moments(want=("J",))
        groups, tables = g.sweep_plan()["groups"], g.sweep_table()["bytes"]
    least = groups * N * ts * 10 + 128 * N + tables + (8 * 13 + 8 * 17 if prec == "mixed" else 8 * 11) * N
    assert rt.grid_footprint(p, prec) >= least


def test_only_grids_that_stream_count_a_table(rt):
    """A second-order request holds no table (2 x 4 bytes per ray and cell, 2 x 8 of the
    FP64 iterations' grid), nor does a subdomain (2 x 8)."""
    p = W.random_box(32, 32, 32, seed=610, n_mu=8, eps_range=(0.3, 1.0))
    N, na = p.chi.size, 80
    srv = rt.Server(workers=1)
    fp = {}
    for interp in ("linear", "quadratic"):
        i = srv.submit(p, prec="mixed", interp=interp, tol=1e-3)
        fp[interp] = srv.wait(i)["footprint"]
        srv.fetch(i)
    srv.close()
    assert fp["linear"] == rt.grid_footprint(p)
    assert fp["quadratic"] <= fp["linear"] - 0.95 * 24 * na * N
    q = W.random_box(32, 32, 32, seed=610, n_mu=8, bc_lo=(P, P, X), bc_hi=(P, P, X))
    r = W.random_box(32, 32, 32, seed=610, n_mu=8, bc_lo=(P, P, T), bc_hi=(P, P, V))
    assert rt.grid_footprint(q, "fp64") <= rt.grid_footprint(r, "fp64") - 0.95 * 16 * na * N
