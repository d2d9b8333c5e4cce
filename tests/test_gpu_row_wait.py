"""A streamed sweep whose wait on a neighbouring strip's edge row runs out (a poll limit
of 0: no wait is granted one) ends by itself with device error code 33, in the planes of
two strips and of sixteen, with many more planes than a word's byte count would hold
unanswered; the grid then solves as a fresh one."""
import numpy as np
import pytest

from paper_1201_2222_gb300 import workloads as W

torch = pytest.importorskip("torch")
pytestmark = pytest.mark.gpu

P, V, T = 0, 1, 2


@pytest.fixture(scope="module")
def rt():
    if not torch.cuda.is_available():
        pytest.skip("no CUDA device")
    from paper_1201_2222_gb300 import build, rt as _rt
    build.build()
    return _rt


def _grid(rt, p, prec, **cfg):
    g = rt.Grid.from_problem(p, prec=prec)
    g.set_sweep_config(**cfg)
    g.set_opacity_source(p.chi, p.eps, p.B, p.freq_w)
    return g


@pytest.mark.parametrize("prec", ["fp64", "mixed"])
@pytest.mark.parametrize("shape,strips", [((24, 20, 12), 2), ((17, 9, 16), 9), ((64, 16, 512), 16)])
def test_a_wait_that_runs_out(rt, prec, shape, strips):
    p = W.random_box(*shape, seed=520, n_mu=6, bc_lo=(P, P, T), bc_hi=(P, P, V))
    cfg = dict(cluster_ctas=strips, variant=3)
    with _grid(rt, p, prec, **cfg) as g:
        g.set_row_wait_limit(0)
        with pytest.raises(rt.RTError) as e:
            g.formal_solve(p.B)
        assert e.value.status == rt.RT_ERR_CUDA and "code 33" in str(e.value)
        with pytest.raises(rt.RTError) as e:
            g.ali_solve(tol=1e-6, max_iter=20)
        assert e.value.status == rt.RT_ERR_CUDA and "code 33" in str(e.value)
        assert g.sweep_table()["streams"]
        g.set_row_wait_limit(1 << 20)
        a = g.ali_solve(tol=1e-6, max_iter=400, raise_on_fail=False)
        with _grid(rt, p, prec, **cfg) as fresh:
            assert fresh.ali_solve(tol=1e-6, max_iter=400, raise_on_fail=False) == a
            np.testing.assert_array_equal(g.get_S(), fresh.get_S())
        with pytest.raises(rt.RTError) as e:
            g.set_row_wait_limit(-1)
        assert e.value.status == rt.RT_ERR_ARG


def test_a_lost_row_of_a_formal_solution_on_a_stream_is_reported_later(rt):
    p = W.random_box(24, 20, 12, seed=530, n_mu=6, bc_lo=(P, P, T), bc_hi=(P, P, V))
    with _grid(rt, p, "fp64", cluster_ctas=4, variant=3) as g:
        g.set_row_wait_limit(0)
        B = torch.from_numpy(p.B).cuda()
        torch.cuda.synchronize()
        with torch.cuda.stream(torch.cuda.Stream()):
            g.formal_solve(B)                               # returns without reading the state
        g.set_row_wait_limit(1 << 20)
        with pytest.raises(rt.RTError) as e:
            g.ali_solve(tol=1e-6, max_iter=20)
        assert e.value.status == rt.RT_ERR_CUDA and "code 33" in str(e.value)
        g.ali_solve(tol=1e-6, max_iter=20, raise_on_fail=False)


def test_a_lost_row_of_the_fp64_iterations_is_reported(rt):
    """A solve of one iteration, which a mixed grid does on its internal FP64 grid (planes
    of 96 x 96 cells, several strips)."""
    p = W.random_box(96, 96, 96, seed=540, n_mu=6, bc_lo=(P, P, T), bc_hi=(P, P, V))
    with _grid(rt, p, "mixed") as g:
        g.set_row_wait_limit(0)
        with pytest.raises(rt.RTError) as e:
            g.ali_solve(tol=1e-6, max_iter=1)
        assert e.value.status == rt.RT_ERR_CUDA and "code 33" in str(e.value)
        g.set_row_wait_limit(1 << 20)
        it, _, st = g.ali_solve(tol=1e-6, max_iter=1, raise_on_fail=False)
        assert it == 1 and st == rt.RT_ERR_NOT_CONVERGED


def test_a_stepped_solve_that_lost_a_row_must_begin_again(rt):
    p = W.random_box(24, 20, 12, seed=550, n_mu=6, bc_lo=(P, P, T), bc_hi=(P, P, V))
    with _grid(rt, p, "fp64", cluster_ctas=4, variant=3) as g:
        g.ali_begin()
        g.ali_iterate(2)
        g.set_row_wait_limit(0)
        with pytest.raises(rt.RTError) as e:
            g.ali_iterate(2)
        assert e.value.status == rt.RT_ERR_CUDA and "code 33" in str(e.value)
        g.set_row_wait_limit(1 << 20)
        with pytest.raises(rt.RTError) as e:
            g.ali_iterate(2)
        assert e.value.status == rt.RT_ERR_STATE
        g.ali_begin()
        a = g.ali_iterate(3)
        with _grid(rt, p, "fp64", cluster_ctas=4, variant=3) as fresh:
            fresh.ali_begin()
            assert fresh.ali_iterate(3) == a
            np.testing.assert_array_equal(g.get_S(), fresh.get_S())
