"""min_p and min_rho of the norms for states that blow up: the quotient |m|^2 / rho at a density of zero, at
infinite or overflowing momenta and at the ends of the range has to come out as the division gives it."""
import numpy as np
import pytest

from paper_2306_06744_gb300 import fr
from paper_2306_06744_gb300 import workloads as W

pytestmark = pytest.mark.gpu


@pytest.mark.parametrize("name", ["vortex2d_p2_small", "vortex3d_p2_tube"])
@pytest.mark.parametrize("rho,m", [(0.0, 1.0), (-0.0, 1.0), (0.0, 0.0), (1.0, np.inf), (1.0, -np.inf), (1.0, 1e200),
                                   (1.0, np.nan), (np.nan, 1.0), (np.inf, 1.0), (4e-310, 1.0), (4e-310, 1e-160),
                                   (1e308, 1.3e154), (1e-300, 1e10), (-1.0, 3.0)])
def test_min_pressure_as_the_division_gives_it(name, rho, m):
    cfg = W.config(name)
    cfg.update(Dbase=2, Dmax=3, init_passes=0, indicator=2, dt=1e-3)
    g = fr.Mesh(cfg)
    u = g.state().copy()
    dim = cfg["dim"]
    u[5, 0, 3], u[5, dim, 3] = rho, m
    g.set_state(g.leaves(), u)
    with np.errstate(all="ignore"):
        m2 = (u[:, 1:1 + dim] ** 2).sum(1)
        p = (cfg["gamma"] - 1.0) * (u[:, -1] - 0.5 * m2 / u[:, 0])
    n = g.norms()
    assert n["min_rho"] == np.fmin.reduce(u[:, 0].ravel())
    want = np.fmin.reduce(p.ravel())
    # 2 dim + 4 roundings, each 2^-53 of E or of the kinetic energy, at the point of the minimum
    if np.isinf(want):
        assert n["min_p"] == want
    else:
        assert abs(n["min_p"] - want) <= 20 * 2.0 ** -53 * (np.abs(want) + 10.0)
