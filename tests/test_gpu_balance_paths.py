"""Paths of the 2:1 balance that depend on how many octants a pass generates."""
import ctypes as C

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


class _Limited:
    """torch's caching allocator behind a limit of the bytes held at a time and a range of block sizes that
    are refused (the host's refusal: NULL, as when the device is full)."""

    def __init__(self, limit=1 << 62, refuse=(0, 0)):
        import torch
        dev = torch.cuda.current_device()
        self.held, self.peak, self.refused = {}, 0, 0

        def alloc(nbytes, stream, ctx):
            if sum(self.held.values()) + nbytes > limit or refuse[0] <= nbytes < refuse[1]:
                self.refused += 1
                return None
            p = torch.cuda.caching_allocator_alloc(int(nbytes), dev, int(stream or 0))
            self.held[p] = nbytes
            self.peak = max(self.peak, sum(self.held.values()))
            return p

        def free(ptr, stream, ctx):
            del self.held[ptr]
            torch.cuda.caching_allocator_delete(int(ptr))

        self._keep = fr.ALLOC_FN(alloc), fr.FREE_FN(free)
        self.struct = fr.FRAllocator(*self._keep, None)


def _balance(dim, Dmax, keys, alloc):
    import torch
    k = torch.from_numpy(keys.view(np.int64)).cuda()
    out = torch.empty(8 * len(keys), dtype=torch.int64, device="cuda")
    n = C.c_int64()
    rc = fr.load().fr_tree_balance_alloc(dim, Dmax, C.c_void_p(k.data_ptr()), len(keys), C.c_void_p(out.data_ptr()),
                                         out.numel(), C.byref(n), C.c_void_p(torch.cuda.current_stream().cuda_stream),
                                         C.byref(alloc.struct))
    assert not alloc.held, "scratch not returned"
    return rc, out[:n.value].cpu().numpy().view(np.uint64) if rc == 0 else None


def test_balance_in_little_memory():
    # 2^18 leaves of one depth (nothing to split): 9 MB is what a call needs whose released blocks go back
    # at once and whose passes have room for 2n octants (8.65 MB)
    d, Dmax = 6, 8
    x = np.stack(np.meshgrid(*[np.arange(1 << d)] * 3, indexing="ij"), -1).reshape(-1, 3) << (Dmax - d)
    keys = np.sort(O.morton_encode(3, Dmax, np.concatenate([np.full((len(x), 1), d), x], 1).astype(np.int32)))
    free = _Limited()
    rc, got = _balance(3, Dmax, keys, free)
    assert rc == 0 and np.array_equal(got, keys) and free.peak > 9_000_000
    tight = _Limited(limit=9_000_000)
    rc, got = _balance(3, Dmax, keys, tight)
    assert rc == 0 and tight.refused > 0 and np.array_equal(got, keys)
    rc, _ = _balance(3, Dmax, keys, _Limited(limit=2_000_000))
    assert rc == fr.FR_ENOMEM


def test_balance_whose_octants_outgrow_the_room():
    # a strip of 2^15 leaves of depth 16 beside a depth-1 leaf: its first pass generates more than 2n octants
    # and less than 8n; where the larger room is refused they are counted and generated at exact positions
    Dmax = 16
    X0 = 1 << (Dmax - 1)
    boxes, stack = [(1, X0, 0, 0), (1, 0, X0, 0), (1, X0, X0, 0)], [(1, 0, 0)]
    while stack:
        d, x, y = stack.pop()
        w = 1 << (Dmax - d)
        if x + w == X0 and d < Dmax:
            stack += [(d + 1, x + (c & 1) * (w // 2), y + (c >> 1) * (w // 2)) for c in range(4)]
        else:
            boxes.append((d, x, y, 0))
    keys = np.sort(O.morton_encode(2, Dmax, np.array(boxes, dtype=np.int32)))
    want = O.balance(2, Dmax, keys)
    room = len(keys) * 8 * 8 * 5 // 4  # bytes of 8n octants with the buffers' slack; blocks round up by 1/8
    launches = []
    for alloc in (_Limited(), _Limited(refuse=(room, room * 9 // 8 + 4096))):
        n0 = fr.kernel_launches()
        rc, got = _balance(2, Dmax, keys, alloc)
        launches.append(fr.kernel_launches() - n0)
        assert rc == 0 and np.array_equal(got, want)
    assert alloc.refused > 0 and launches[1] > launches[0]
