"""Psi0 of float32 sweeps.  A single bright cell in a dark uniform medium: every ray's
S and I upwind of it are 0, so its J is the mean of Psi0(chi s) over the rays.  With
spacings equal to the direction cosines s is 1 and the upwind point a cell centre, so
that dtau is chi exactly; one ray a group, whose partials are summed exactly.

The series evaluated by Horner's rule with x < 1/2: the last subtraction, of a value
of 0.42 to 0.5, rounds by 3e-8 / 0.42, the last product by 6e-8, the terms before
them by less than 2e-8 together: 1.5e-7 at most, without a preferred sign."""
import numpy as np
import pytest

from paper_1201_2222_gb300 import workloads as W

torch = pytest.importorskip("torch")
pytestmark = pytest.mark.gpu

V = 1


def psi0(x):
    """sum_{n >= 1} (-1)^(n + 1) x^n / (n + 1)!"""
    x = x.astype(np.longdouble)
    s, term = np.zeros_like(x), np.ones_like(x)
    for n in range(1, 25):
        term = term * x / (n + 1)
        s += term if n % 2 else -term
    return s


@pytest.mark.parametrize("nx,ny,moments", [(5, 3, False), (5, 3, True), (8, 4, False), (8, 4, True)])
def test_thin_cells(nx, ny, moments):
    from paper_1201_2222_gb300 import build, rt
    if not torch.cuda.is_available():
        pytest.skip("no CUDA device")
    build.build()
    nf, nz, at = 512, 3, (1, 1, 2)
    tau = np.exp(np.linspace(np.log(1e-6), np.log(0.499), nf)).astype(np.float32).astype(np.float64)
    chi = np.broadcast_to(tau[:, None, None, None], (nf, nz, ny, nx)).copy()
    h = 1 / np.sqrt(3.0)
    p = W.Problem(name="bright cell", nx=nx, ny=ny, nz=nz, n_mu=2, chi=chi, eps=np.full_like(chi, 0.5),
                  B=np.zeros_like(chi), freq_w=np.ones(nf), bc_lo=(V, V, V), bc_hi=(V, V, V), dx=h, dy=h, dz=h)
    S = np.zeros_like(chi)
    S[(slice(None),) + at] = 1.0
    with rt.Grid.from_problem(p, prec="mixed") as g:
        g.set_sweep_config(angles_per_group=1)
        g.set_opacity_source(p.chi, p.eps, p.B, p.freq_w)
        J = g.formal_solve(S)
        if moments:
            J = g.moments(want=("J",))["J"]
        assert g.sweep_table()["streams"]
    err = (J[(slice(None),) + at] / psi0(tau) - 1).astype(float)
    assert np.max(np.abs(err)) < 1.5e-7
    assert abs(np.mean(err)) < 2e-8
