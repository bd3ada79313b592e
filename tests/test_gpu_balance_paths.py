"""Paths of the 2:1 balance that depend on how many octants a pass generates."""
import numpy as np
import pytest

import oracle as O
from paper_2306_06744_gb300 import fr
from paper_2306_06744_gb300 import workloads as W

pytestmark = pytest.mark.gpu


def _circle_tree(Dbase, Dmax):
    """Balanced quadtree of depth Dmax - 1 along a circle."""
    side = 1 << Dmax
    c, r = side * 0.5, side * 0.31
    work = [(Dbase, x * (side >> Dbase), y * (side >> Dbase)) for x in range(1 << Dbase) for y in range(1 << Dbase)]
    out = []
    while work:
        nxt = []
        for d, x, y in work:
            w = side >> d
            if d < Dmax - 1 and abs(np.hypot(x + w / 2 - c, y + w / 2 - c) - r) < 0.75 * w:
                nxt += [(d + 1, x + a * w // 2, y + b * w // 2) for a in (0, 1) for b in (0, 1)]
            else:
                out.append((d, x, y, 0))
        work = nxt
    return O.balance(2, Dmax, np.sort(O.morton_encode(2, Dmax, np.array(out, dtype=np.int32))))


def test_an_adaptation_takes_the_same_path_on_every_run():
    # flags around the number at which the deepest balance pass outgrows the 4096 octants of an adaptation
    # issued without synchronisation: whether it does must not change from run to run
    Dbase, Dmax = 3, 11
    keys = _circle_tree(Dbase, Dmax)
    deep = O.morton_decode(2, Dmax, keys)[:, 0] == Dmax - 1
    assert len(keys) == 13156 and deep.sum() == 5840
    g = fr.Mesh(dict(W.config("vortex2d_p2_small"), p=1, Dbase=Dbase, Dmax=Dmax, init_passes=0, indicator=2, dt=1e-3))
    u = np.ones((len(keys), 4, 4))
    u[:, 3] = 2.5
    r = W.random_uniform(len(keys), 7)
    seen = set()
    for q in np.arange(0.115, 0.128, 0.0004):
        flags = (deep & (r < q)).astype(np.int8)
        paths = set()
        for _ in range(8):
            g.set_state(keys, u)
            paths.add(g.adapt(flags, stats=True)["balance_exact_depth"])
        assert len(paths) == 1, (q, paths)
        seen |= paths
    assert seen == {0, Dmax}  # both sides of the limit were met
