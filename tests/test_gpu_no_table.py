"""Solves without a table of segment weights (rt_set_table_limit 0): the kernels that
grids take where the table has no room -- the float32 and FP64 pipelined sweeps, the
FP64 sweep of one cell per thread, their shared launches -- replanned at a grid's first
solve.  Against the oracle; tolerances as in test_gpu_parity and test_gpu_stream
(rounding only: 1e-10 FP64, 1e-5 float32)."""
import contextlib

import numpy as np
import pytest

from oracle import oracle as O
from paper_1201_2222_gb300 import workloads as W

torch = pytest.importorskip("torch")
pytestmark = pytest.mark.gpu

P, V, T = 0, 1, 2

CASES = [   # nx, ny, nz, n_mu, bc_lo, bc_hi, precision, sweep config
    (32, 16, 12, 6, (P, P, T), (P, P, V), "mixed", {}),                                # whole 16-byte rows
    (36, 40, 33, 4, (T, V, P), (V, T, P), "mixed", dict(angles_per_group=3, cluster_ctas=4, variant=3)),
    (30, 31, 29, 4, (P, P, P), (P, P, P), "mixed", dict(angles_per_group=2, cluster_ctas=2)),
    (20, 24, 1, 6, (P, T, P), (P, V, P), "mixed", {}),
    (18, 14, 10, 4, (P, P, T), (P, P, V), "fp64", {}),
    (17, 12, 16, 4, (P, P, P), (P, P, P), "fp64", dict(angles_per_group=2, cluster_ctas=2, variant=3)),
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


@contextlib.contextmanager
def free_memory_of(nbytes):
    """The device's free memory cut down to nbytes."""
    torch.cuda.empty_cache()
    hold = torch.empty(torch.cuda.mem_get_info()[0] - nbytes, dtype=torch.uint8, device="cuda")
    try:
        yield
    finally:
        del hold
        torch.cuda.empty_cache()


def _grid(rt, p, prec, cfg, limit=0, scheme="jacobi"):
    g = rt.Grid.from_problem(p, prec=prec)
    if cfg:
        g.set_sweep_config(**cfg)
    g.set_iteration(scheme)
    g.set_opacity_source(p.chi, p.eps, p.B, p.freq_w)
    if limit is not None:
        g.set_table_limit(limit)
    return g


@pytest.mark.parametrize("case", range(len(CASES)))
def test_formal_solutions_iterations_and_moments(rt, case):
    nx, ny, nz, n_mu, lo, hi, prec, cfg = CASES[case]
    p = W.random_box(nx, ny, nz, seed=400 + case, n_mu=n_mu, nf=2 if case % 2 else 1, bc_lo=lo, bc_hi=hi)
    og = O.Grid.from_problem(p)
    tol = 1e-10 if prec == "fp64" else 1e-5
    with _grid(rt, p, prec, cfg) as g:
        S = np.random.default_rng(case).uniform(0.3, 2.0, p.chi.shape)
        G = [O.init_ghosts(og, S[f]) for f in range(p.nf)]
        for k in range(3):                       # the later ones from lagged periodic ghosts
            J = g.formal_solve(S if k == 0 else None)
            assert g.sweep_table() == {"streams": False, "bytes": 0}
            for f in range(p.nf):
                ref = O.formal_solution(og, p.chi[f], S[f], p.B[f], G_prev=G[f])
                G[f] = ref["G_next"]
                assert rel(J[f], ref["J"]) < tol
        it, _, _ = g.ali_solve(tol=1e-6, max_iter=60, raise_on_fail=False)
        ref = O.ali_solve(og, p.chi, p.eps, p.B, p.freq_w, tol=1e-6, max_iter=60)
        m = g.moments()
        assert it == ref["iters"]
        assert rel(g.get_S(), ref["S"]) < tol
        assert rel(m["J"], ref["J"]) < tol
        assert rel(m["K"][:, :3], ref["K"][:, :3]) < tol
        assert g.sweep_table() == {"streams": False, "bytes": 0}
        # and with the table again
        g.set_table_limit(-1)
        it, _, _ = g.ali_solve(tol=1e-6, max_iter=60, raise_on_fail=False)
        assert it == ref["iters"] and rel(g.get_S(), ref["S"]) < tol
        t = g.sweep_table()
        assert t["streams"] and t["bytes"] > 0


@pytest.mark.parametrize("prec,shape,cfg", [("mixed", (256, 256, 16), dict(angles_per_group=3, cluster_ctas=16)),
                                            ("fp64", (128, 128, 16), dict(angles_per_group=2, cluster_ctas=6))])
def test_a_plan_that_only_the_streamed_sweep_fits(rt, prec, shape, cfg):
    """Such rays and strips (the pipelined sweep would need 238 and 268 KB of shared
    memory a CTA for them) are set aside when the table has no room, and taken again
    when it has; asked for without the room they are an error that leaves the grid
    as it was."""
    p = W.random_box(*shape, seed=430, n_mu=6, bc_lo=(P, P, T), bc_hi=(P, P, V))
    ref = O.formal_solution(O.Grid.from_problem(p), p.chi[0], p.B[0], p.B[0], nthreads=O.max_threads())["J"]
    tol = 1e-10 if prec == "fp64" else 1e-5
    with _grid(rt, p, prec, dict(cfg, variant=3)) as g:
        plan = lambda: (g.sweep_plan()["rays_per_group"], g.sweep_plan()["cluster"])
        assert plan() == tuple(cfg.values())
        assert rel(g.formal_solve(p.B)[0], ref) < tol
        assert not g.sweep_table()["streams"] and plan() != tuple(cfg.values())
        with pytest.raises(rt.RTError) as e:
            g.set_sweep_config(**cfg, variant=3)
        assert e.value.status == rt.RT_ERR_ARG
        assert rel(g.formal_solve(p.B)[0], ref) < tol
        g.set_table_limit(-1)
        assert rel(g.formal_solve(p.B)[0], ref) < tol
        assert g.sweep_table()["streams"] and plan() == tuple(cfg.values())


@pytest.mark.parametrize("first", [None, 0])
def test_tuned_plans_are_not_shared_with_grids_that_have_a_table(rt, first):
    """The cache answers a second grid of the same kind, and no grid of the other."""
    p = W.random_box(24, 20, 16 if first is None else 18, seed=440, n_mu=2)
    tuned = {}
    for limit in (first, -1 if first == 0 else 0):
        for again in range(2):
            with _grid(rt, p, "mixed", {}, limit) as g:
                plan, n = g.autotune(), g.stats()["kernel_launches"]
                J = g.formal_solve(p.B)
                assert limit != 0 or not g.sweep_table()["streams"]
                assert (n < 50) == bool(again), n        # a search launches hundreds of kernels
                assert tuned.setdefault(limit, plan) == plan
                np.testing.assert_allclose(J, tuned.setdefault("J", J), rtol=1e-5)


def test_fp64_table_takes_the_memory_there_is(rt):
    """A table of 0.68 GB in 1.2 GB of free memory."""
    p = W.random_box(96, 96, 96, seed=450, n_mu=6)
    with _grid(rt, p, "fp64", {}, None) as g:
        with free_memory_of(1200 << 20):
            J = g.formal_solve(p.B)
            t = g.sweep_table()
        assert t == {"streams": True, "bytes": 2 * 48 * 96 ** 3 * 8}
        np.testing.assert_array_equal(J, g.formal_solve(p.B))


@pytest.mark.parametrize("prec", ["fp64", "mixed"])
def test_a_later_medium_finds_the_room_that_an_earlier_one_had_not(rt, prec):
    """A table of 0.27 GB (0.13 in float32) when 0.2 GB are free, and when all are."""
    p = W.random_box(128, 128, 128, seed=470, n_mu=2)
    with _grid(rt, p, prec, {}, None) as g:
        with free_memory_of(200 << 20):
            J = g.formal_solve(p.B)
            assert g.sweep_table() == {"streams": False, "bytes": 0}
        g.set_opacity_source(p.chi, p.eps, p.B, p.freq_w)
        J2 = g.formal_solve(p.B)
        assert g.sweep_table()["streams"]
    np.testing.assert_allclose(J2, J, rtol=1e-12 if prec == "fp64" else 1e-5)


def test_tables_give_way_to_what_the_moments_need(rt):
    """With 1.16 GB free and no table but the FP64 iterations' (0.27 GB) the moments'
    0.87 GB fit; a float32 table of 0.13 GB must not take their place."""
    p = W.random_box(128, 128, 128, seed=490, n_mu=2)
    with _grid(rt, p, "mixed", dict(angles_per_group=1), None) as g:
        g.ali_solve(tol=1e-6, max_iter=5, raise_on_fail=False)
        want = g.moments(want=("J", "K"))
    with _grid(rt, p, "mixed", dict(angles_per_group=1), None) as g:
        with free_memory_of(1160 << 20):
            g.ali_solve(tol=1e-6, max_iter=5, raise_on_fail=False)
            assert g.sweep_table()["bytes"] == (8 + 16) * 8 * 128 ** 3
            got = g.moments(want=("J", "K"))
            assert g.sweep_table()["bytes"] == 0
            g.ali_solve(tol=1e-6, max_iter=5, raise_on_fail=False)
            again = g.moments(want=("J", "K"))
    for m in (got, again):
        assert rel(m["J"], want["J"]) < 1e-5 and rel(m["K"][:, :3], want["K"][:, :3]) < 1e-5


@pytest.mark.parametrize("prec", ["fp64", "mixed"])
def test_second_order_holds_no_table(rt, prec):
    p = W.random_box(16, 12, 8, seed=480, n_mu=4)
    with _grid(rt, p, prec, {}, None) as g:
        a = g.ali_solve(tol=1e-6, max_iter=200)[0], g.get_S()
        assert g.sweep_table()["bytes"] > 0
        g.set_interpolation("quadratic")
        assert g.sweep_table()["bytes"] == 0
        g.ali_solve(tol=1e-6, max_iter=20, raise_on_fail=False)
        assert g.sweep_table()["bytes"] == 0
        g.set_interpolation("linear")
        b = g.ali_solve(tol=1e-6, max_iter=200)[0], g.get_S()
        assert a[0] == b[0] and g.sweep_table()["bytes"] > 0
        np.testing.assert_array_equal(a[1], b[1])


def test_fp64_tables_of_unpadded_rows(rt):
    """Rows of one cell: the streamed sweep's table (rows padded to 16 bytes) is twice
    as large as the one-cell-per-thread sweep's, which fits the limit alone."""
    p = W.random_box(1, 30, 20, seed=460, n_mu=4, bc_lo=(P, P, T), bc_hi=(P, P, V))
    ref = O.formal_solution(O.Grid.from_problem(p), p.chi[0], p.B[0], p.B[0])["J"]
    small = 2 * 24 * 30 * 20 * 8
    with _grid(rt, p, "fp64", {}, small) as g:
        assert rel(g.formal_solve(p.B)[0], ref) < 1e-10
        assert g.sweep_table() == {"streams": False, "bytes": small}


@pytest.mark.parametrize("prec", ["fp64", "mixed"])
def test_gauss_seidel(rt, prec):
    """One iteration (the forward phase by the sweep, S by the reverse phase)."""
    p = W.random_box(20, 12, 16, seed=420, n_mu=4, bc_lo=(P, P, T), bc_hi=(P, P, V))
    og = O.Grid.from_problem(p)
    ref = O.ali_solve(og, p.chi, p.eps, p.B, p.freq_w, tol=0.0, max_iter=1, moments=False, method="gauss_seidel")
    with _grid(rt, p, prec, {}, scheme="gauss_seidel") as g:
        g.ali_solve(tol=0.0, max_iter=1, raise_on_fail=False)
        assert not g.sweep_table()["streams"]
        assert rel(g.get_S(), ref["S"]) < (1e-10 if prec == "fp64" else 1e-5)


def test_lock_step_equals_each_alone_bit_for_bit(rt):
    """Grids with and without a table, of both precisions, in one set."""
    probs = [(W.stratified_atmosphere(16, nxy=8), "mixed", 0), (W.turbulent_box(24, n_mu=8), "mixed", 0),
             (W.random_box(12, 8, 10, seed=71, n_mu=6, bc_lo=(T, P, V), bc_hi=(V, P, T)), "mixed", None),
             (W.stratified_atmosphere(12, nxy=4, eps=1e-3), "mixed", None),
             (W.random_box(8, 8, 8, seed=72, n_mu=4), "fp64", 0), (W.random_box(8, 12, 6, seed=75, n_mu=6), "fp64", 0),
             (W.random_box(9, 7, 6, seed=73, n_mu=4), "mixed", 0), (W.random_box(7, 9, 6, seed=74, n_mu=4), "mixed", 0)]
    cfg = dict(cluster_ctas=2, variant=3)
    alone = []
    for p, prec, limit in probs:
        with _grid(rt, p, prec, cfg, limit) as g:
            it, _, _ = g.ali_solve(tol=1e-6, max_iter=5000)
            alone.append((it, g.get_S()))
    grids = [_grid(rt, p, prec, cfg, limit) for p, prec, limit in probs]
    out = rt.ali_solve_many(grids, tol=1e-6, max_iter=5000)
    for g, (it, _, _), (it1, S1), (p, prec, limit) in zip(grids, out, alone, probs):
        assert it == it1
        np.testing.assert_array_equal(g.get_S(), S1)
        assert g.sweep_table()["streams"] == (limit is None)
        assert g.stats()["shared_launches"] > 0          # each has a partner of its kind
        g.close()


def test_bad_limits_are_errors(rt):
    with rt.Grid(4, 4, 4) as g:
        with pytest.raises(rt.RTError) as e:
            g.set_table_limit(-2)
        assert e.value.status == rt.RT_ERR_ARG
