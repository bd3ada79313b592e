"""Residuals of the FP64 form for states whose interface flux its integer products could get wrong.  The
states are constant in every element of a uniform mesh, so the method reduces to
R = -sum_a (2/h) [g'_L (F_- - f) + g'_R (F_+ - f)], evaluated here in numpy FP64 with the Rusanov flux's wave
speed as fmax gives it (one that is not a number loses to one that is)."""
import numpy as np
import pytest

import oracle as O
from paper_2306_06744_gb300 import fr
from paper_2306_06744_gb300 import workloads as W

pytestmark = pytest.mark.gpu

GAMMA = 1.4


def _mesh(dim, p, depth):
    cfg = dict(W.config("vortex2d_p2_small" if dim == 2 else "vortex3d_p2_tube"), dim=dim, p=p, L=8.0, Dbase=depth,
               Dmax=depth + 1, init_passes=0, indicator=2, dt=1e-3)
    g = fr.Mesh(cfg)
    return g, g.leaves(), O.morton_decode(dim, depth + 1, g.leaves())[:, 1:1 + dim] // 2


def _flux(q, a):
    dim = q.shape[1] - 2
    v = q[:, 1 + a] / q[:, 0]
    ke = 0.5 * (q[:, 1:1 + dim] ** 2).sum(1) / q[:, 0]
    p = (GAMMA - 1.0) * (q[:, -1] - ke)
    f = q * v[:, None]
    f[:, 1 + a] += p
    f[:, -1] += p * v
    return f, np.abs(v) + np.sqrt(GAMMA * p / q[:, 0]), np.abs(v), (GAMMA - 1.0) * (np.abs(q[:, -1]) + ke)


def _rhs(q, cells, p, depth):
    """R [M][nv][N] of element-constant states q [M][nv], and the size of the terms it is formed from."""
    dim, n, h = q.shape[1] - 2, p + 1, 8.0 / 2 ** depth
    o = O.operators(p)
    index = {tuple(c): e for e, c in enumerate(cells)}
    R = np.zeros((len(q), dim + 2) + (n,) * dim)
    S = np.zeros((len(q), dim + 2))
    tr = np.where(np.isinf(q), np.nan, q)  # traces: the weights have both signs, so inf - inf
    with np.errstate(all="ignore"):
        for a in range(dim):
            nb = np.array([index[tuple((c + (np.arange(dim) == a)) % 2 ** depth)] for c in cells])
            fe = _flux(q, a)[0]
            f, s, av, pa = _flux(tr, a)
            lam, top = np.fmax(s, s[nb]), np.fmax(np.fmax(s, s[nb]), np.fmax(av, av[nb]))
            F = 0.5 * (f + f[nb] - lam[:, None] * (tr[nb] - tr))
            mag = np.abs(q) + np.abs(q[nb])
            mag[:, 1:1 + dim] = mag[:, 1:1 + dim].max(1, keepdims=True)
            t = top[:, None] * mag + (pa + pa[nb])[:, None]
            t[:, -1] += top * (pa + pa[nb])
            Fm = np.empty_like(F)
            Fm[nb] = F
            T = t.copy()
            T[nb] = np.maximum(T[nb], t)
            S += T
            line = np.zeros((len(q), dim + 2, n))
            line += (Fm - fe)[:, :, None] * o["gL"] + (F - fe)[:, :, None] * o["gR"]
            shape = [len(q), dim + 2] + [1] * dim
            shape[2 + dim - 1 - a] = n
            R -= 2.0 / h * line.reshape(shape)
    return R.reshape(len(q), dim + 2, -1), S * 2.0 / h * max(np.abs(o["gL"]).max(), np.abs(o["gR"]).max())


def _states(M, dim, seed):
    r = W.random_uniform(M * (dim + 2), seed).reshape(M, dim + 2)
    q = np.empty((M, dim + 2))
    q[:, 0] = 0.5 + r[:, 0]
    q[:, 1:1 + dim] = q[:, :1] * (2.0 * r[:, 1:1 + dim] - 1.0)
    q[:, -1] = (0.3 + r[:, -1]) / (GAMMA - 1.0) + 0.5 * (q[:, 1:1 + dim] ** 2).sum(1) / q[:, 0]
    return q


def _run(g, keys, q):
    N = g.N
    g.set_state(keys, np.repeat(q[:, :, None], N, axis=2).copy())
    return g.rhs()


# flux: (6 kappa + 16) 2^-53 of the terms with kappa <= 11 at these pressures (E + ke over E - ke), on
# each side of the comparison, and the element's sums
TOL = 400 * 2.0 ** -53


@pytest.mark.parametrize("dim,p", [(2, 1), (2, 3), (3, 2)])
def test_negative_pressure_on_one_side(dim, p):
    g, keys, cells = _mesh(dim, p, 2)
    q = _states(len(keys), dim, 3)
    bad = 5
    q[bad, 1:1 + dim] = 40.0 * q[bad, 0] * np.array([1.0, -0.7, 0.4])[:dim]  # past its neighbours' wave speeds
    q[bad, -1] = 0.3 * 0.5 * (q[bad, 1:1 + dim] ** 2).sum() / q[bad, 0]
    want, scale = _rhs(q, cells, p, 2)
    got = _run(g, keys, q)
    assert np.isfinite(want).all()
    assert (np.abs(got - want) <= TOL * scale[:, :, None]).all()


@pytest.mark.parametrize("e", [-470, -300, 440])
@pytest.mark.parametrize("dim,p", [(2, 2), (3, 3)])
def test_units_far_from_one(dim, p, e):
    g, keys, cells = _mesh(dim, p, 2)
    q = np.ldexp(_states(len(keys), dim, 8), e)
    want, scale = _rhs(q, cells, p, 2)
    assert (np.abs(_run(g, keys, q) - want) <= TOL * scale[:, :, None]).all()


@pytest.mark.parametrize("jump", [1e2, 1e4, 1e6, 1e8])
@pytest.mark.parametrize("dim,p", [(2, 1), (2, 3), (3, 2)])
def test_density_jump_across_faces(dim, p, jump):
    # one element in eight lighter by the factor, speeds and temperatures alike
    g, keys, cells = _mesh(dim, p, 2)
    q = _states(len(keys), dim, 6)
    q[(cells % 2 == 0).all(1)] /= jump
    want, scale = _rhs(q, cells, p, 2)
    assert (np.abs(_run(g, keys, q) - want) <= TOL * scale[:, :, None]).all()


@pytest.mark.parametrize("value", [np.nan, -np.nan, np.inf, -np.inf])
@pytest.mark.parametrize("dim,p", [(2, 2), (3, 1)])
def test_special_values_reach_the_neighbours(dim, p, value):
    # non-finite wherever the FP64 formula is; elsewhere only in the element and its face neighbours
    depth = 2
    g, keys, cells = _mesh(dim, p, depth)
    ok = _states(len(keys), dim, 4)
    e = 9
    d = np.abs(cells - cells[e])
    near = np.minimum(d, 2 ** depth - d).sum(1) <= 1
    for v in range(dim + 2):
        q = ok.copy()
        q[e, v] = np.copysign(value, -1.0) if np.signbit(value) else value
        want, scale = _rhs(q, cells, p, depth)
        got = _run(g, keys, q)
        assert not np.isfinite(got[~np.isfinite(want)]).any(), v
        assert (np.abs(got - want) <= TOL * scale[:, :, None])[~near].all(), v
