"""Device memory from a caller's allocator that is aligned to 8 bytes only: the common fluxes of the FP32 and
double-word forms are then copied a value at a time instead of 16 bytes at a time (in grids below and above
the size at which the copy starts early).  Same arithmetic, so the same bits."""
import numpy as np
import pytest

from paper_2306_06744_gb300 import fr
from paper_2306_06744_gb300 import workloads as W

pytestmark = pytest.mark.gpu


class _Shifted(fr._TorchAllocator):
    def __init__(self, device):
        super().__init__(device)
        alloc, free = self._a, self._f

        def shifted(nbytes, stream, ctx):
            p = alloc(nbytes + 16, stream, ctx)
            return p + 8 if p else None

        def unshift(ptr, stream, ctx):
            free(ptr - 8 if ptr else None, stream, ctx)

        self._inner = alloc, free
        self._a, self._f = fr.ALLOC_FN(shifted), fr.FREE_FN(unshift)
        self.struct = fr.FRAllocator(self._a, self._f, None)


@pytest.mark.parametrize("precision", [0, 1, 4])
@pytest.mark.parametrize("dim,p,depth", [(2, 1, 4), (2, 2, 4), (2, 3, 4), (3, 1, 3), (3, 2, 2), (3, 3, 2), (3, 4, 2),
                                         (2, 2, 10)])
def test_memory_aligned_to_8_bytes(monkeypatch, dim, p, depth, precision):
    cfg = W.config("vortex2d_p2_small" if dim == 2 else "vortex3d_p2_tube")
    cfg.update(dim=dim, p=p, Dbase=depth, Dmax=depth + 1, precision=precision, init_passes=0, indicator=2, dt=1e-3)
    out = []
    for a in (fr._TorchAllocator, _Shifted):
        monkeypatch.setattr(fr, "_TorchAllocator", a)
        g = fr.Mesh(cfg)
        flags = np.zeros(g.M, dtype=np.int8)
        flags[::7] = 1
        g.adapt(flags)  # hanging faces too
        g.step(2)
        out.append(g.state().copy())
        g.close()
    assert np.isfinite(out[0]).all() and np.array_equal(out[0], out[1])


@pytest.mark.parametrize("precision,bar", [(1, 1e-5), (4, 1e-11)])
def test_early_fetch_agrees_with_the_fp64_form(precision, bar):
    # 75k blocks: the fetch starts before the volume part.  Two steps of dt / h = 0.1 at speeds of O(1): six
    # stages, each off by some tens of roundings (2^-24, 2^-47) of a tenth of the state; a flux that is read
    # too soon is off by its changes, at least 1e-4 of it
    cfg = W.config("vortex2d_p2_small")
    cfg.update(Dbase=10, Dmax=11, init_passes=0, indicator=2, dt=1e-3)
    out = []
    for q in (0, precision):
        g = fr.Mesh(dict(cfg, precision=q))
        g.step(2)
        out.append(g.state().copy())
        g.close()
    assert np.linalg.norm((out[1] - out[0]).ravel()) < bar * np.linalg.norm(out[0].ravel())
