"""The work a user of this framework has it do, as cases that can be timed and compared.

Kinds of case:

``cycle``  one adaptation cycle of a vortex run: keys and state go in from pinned host memory
           (`Mesh.set_state`, also the restart path), 10 SSP-RK3 steps and one adaptation
           (`Mesh.run`), then the norms, keys and state come back to pinned host memory.
``tree``   a 2:1 balanced tree from a cloud of surface points: tree completion, then balance.
``learned`` the learned indicator on a mesh: features, then the MLP's logits and flags.
``train``  one Adam step of the learned indicator on a batch.

`exact` restates the method in plain numpy and torch FP64 (flux reconstruction on nonconforming
trees, density-gradient flags, the adaptation edit, vertex 2:1 balance, interpolation and L2
projection, the MLP and its gradient) and shares no code with the package.
"""
from __future__ import annotations

import math

import numpy as np
import torch

from paper_2306_06744_gb300 import fr

F64 = torch.float64
GAMMA = 1.4


def listed():
    return [
        # the smallest run (paper's small 2D domain, p = 2): launch latency counts
        dict(name="cycle_2d_p2_small_f64", kind="cycle", dim=2, p=2, prec=0, L=10.0, Dbase=4, Dmax=6, nvort=1,
             th_r=0.05, th_c=0.01),
        # the 2D p = 3 run: tens of thousands of elements, about one wave of blocks per kernel
        dict(name="cycle_2d_p3_f64", kind="cycle", dim=2, p=3, prec=0, L=40.0, Dbase=5, Dmax=9, nvort=1,
             th_r=1e-8, th_c=2.5e-9),
        # the lowest degree (the paper's p = 1 rows): little arithmetic per point, most faces per point
        dict(name="cycle_2d_p1_f64", kind="cycle", dim=2, p=1, prec=0, L=40.0, Dbase=5, Dmax=10, nvort=1,
             th_r=1e-7, th_c=2.5e-8),
        # the 3D p = 2 tube
        dict(name="cycle_3d_p2_f64", kind="cycle", dim=3, p=2, prec=0, L=10.0, Dbase=4, Dmax=7, nvort=1,
             th_r=0.03, th_c=0.0075),
        # the four 3D p = 3 tubes at a depth that leaves room for copies of the state: the largest
        dict(name="cycle_3d_p3_f64", kind="cycle", dim=3, p=3, prec=0, L=80.0, Dbase=5, Dmax=8, nvort=4,
             th_r=0.05, th_c=0.0125),
        # the same run in the double-word and the FP32 forms (the faster forms of equal vortex error)
        dict(name="cycle_3d_p3_doubleword", kind="cycle", dim=3, p=3, prec=4, L=80.0, Dbase=5, Dmax=8, nvort=4,
             th_r=0.05, th_c=0.0125),
        dict(name="cycle_3d_p3_f32", kind="cycle", dim=3, p=3, prec=1, L=80.0, Dbase=5, Dmax=8, nvort=4,
             th_r=0.05, th_c=0.0125),
        # 2D p = 3 in the double-word form, the only fast form that keeps this run's error
        dict(name="cycle_2d_p3_doubleword", kind="cycle", dim=2, p=3, prec=4, L=40.0, Dbase=5, Dmax=9, nvort=1,
             th_r=1e-8, th_c=2.5e-9),
        # tree construction from a scanned surface (the paper's first experiment, on a torus)
        dict(name="tree_3d_600k_points", kind="tree", dim=3, n=600000, Dmin=4, Dmax=9),
        # the learned indicator deployed on the 3D p = 3 mesh
        dict(name="learned_3d_p3", kind="learned", dim=3, p=3, M=200000),
        # its training: the default batch, and the large one
        dict(name="train_batch_4096", kind="train", n_in=55, batch=4096),
        dict(name="train_batch_65536", kind="train", n_in=55, batch=65536),
    ]


def draw(rng):
    """Cases of the same ranges: dimension, degree, arithmetic form and depth of a cycle; points
    and depth of a tree; elements of an indicator evaluation; batch and width of a training step."""
    def logint(a, b):
        return int(round(math.exp(rng.uniform(math.log(a), math.log(b)))))

    kind = rng.choice(["cycle", "cycle", "cycle", "cycle", "tree", "learned", "train"])
    if kind == "cycle":
        dim = rng.choice([2, 2, 3])
        L = round(math.exp(rng.uniform(math.log(10.0), math.log(40.0))), 3)
        if dim == 2:
            p = rng.choice([1, 2, 3, 4])
            Dbase = rng.choice([3, 4, 5])
            Dmax = Dbase + rng.choice([1, 2, 3, 4])
            th = 10 ** rng.uniform(-8, -2)
            prec = rng.choice([0, 0, 4])
        else:
            p = rng.choice([1, 2, 3, 4])
            Dbase = 3 if p == 4 else rng.choice([3, 4])
            Dmax = Dbase + rng.choice([1, 2])
            th = 10 ** rng.uniform(-2, -1)
            prec = rng.choice([0, 0, 4, 1])
        th = float("%.3g" % th)
        return dict(kind="cycle", dim=dim, p=p, prec=prec, L=L, Dbase=Dbase, Dmax=Dmax,
                    nvort=1 if L < 20 else rng.choice([1, 2, 4]), th_r=th, th_c=float("%.3g" % (th * 0.25)))
    if kind == "tree":
        return dict(kind="tree", dim=rng.choice([2, 3]), n=logint(1000, 600000), Dmin=rng.choice([2, 3, 4]),
                    Dmax=rng.choice([7, 8, 9]))
    if kind == "learned":
        return dict(kind="learned", dim=rng.choice([2, 3]), p=rng.choice([1, 2, 3, 4]), M=logint(700, 150000))
    return dict(kind="train", n_in=rng.choice([19, 55]), batch=logint(200, 65536))


# ---- plain numpy/torch: operators, trees, vortex ------------------------------------------------

def _lagrange(x, t):
    """l_j(t) for every t (rows) on the nodes x, by products."""
    t = np.atleast_1d(np.asarray(t, dtype=np.float64))
    out = np.ones((t.size, x.size))
    for j in range(x.size):
        for k in range(x.size):
            if k != j:
                out[:, j] *= (t - x[k]) / (x[j] - x[k])
    return out


class _Ops:
    def __init__(self, p):
        n = p + 1
        self.n = n
        x, w = np.polynomial.legendre.leggauss(n)
        D = np.zeros((n, n))
        for i in range(n):
            for j in range(n):
                if i != j:
                    num = np.prod([x[i] - x[k] for k in range(n) if k not in (i, j)])
                    D[i, j] = num / np.prod([x[j] - x[k] for k in range(n) if k != j])
            D[i, i] = -D[i].sum()
        lm, lp = _lagrange(x, -1.0)[0], _lagrange(x, 1.0)[0]
        I = np.stack([_lagrange(x, (x + 2 * h - 1) / 2) for h in (0, 1)])
        P = np.stack([0.5 * (w[None, :] / w[:, None]) * I[h].T for h in (0, 1)])
        self.x, self.w = x, w

        def dev(a):
            return torch.as_tensor(a, dtype=F64, device="cuda")
        self.D, self.lm, self.lp = dev(D), dev(lm), dev(lp)
        self.gL, self.gR = dev(-lm / w), dev(lp / w)
        self.I, self.P, self.wt, self.xt = dev(I), dev(P), dev(w), dev(x)


def _interleave(X, dim):
    """Raw Morton IDs of integer anchors X [.., dim] (torch int64), x in the lowest bit."""
    out = torch.zeros_like(X[..., 0])
    for b in range(20):
        for a in range(dim):
            out |= ((X[..., a] >> b) & 1) << (b * dim + a)
    return out


class _Tree:
    """Leaves as depths d [M] and anchors X [M, dim] in finest units, in Morton order."""

    def __init__(self, dim, Dmax, d, X):
        self.dim, self.Dmax = dim, Dmax
        self.mb = max(1, math.ceil(math.log2(Dmax + 1)))
        key = (_interleave(X, dim) << self.mb) | d
        self.key, o = torch.sort(key)
        self.d, self.X = d[o], X[o]
        self.M = int(d.numel())

    def width(self, d):
        return torch.ones_like(d) << (self.Dmax - d)

    def locate(self, X):
        """Index of the leaf that contains the finest cell at X."""
        return torch.searchsorted(self.key, (_interleave(X, self.dim) << self.mb) | self.Dmax, right=True) - 1


def _children(t, sel):
    """Depths and anchors with the selected leaves replaced by their 2^dim children."""
    nc = 1 << t.dim
    cd = (t.d[sel] + 1).repeat_interleave(nc)
    h = t.width(cd)
    c = torch.arange(nc, device="cuda").repeat(int(sel.sum()))
    off = torch.stack([((c >> a) & 1) * h for a in range(t.dim)], 1)
    return (torch.cat([t.d[~sel], cd]), torch.cat([t.X[~sel], t.X[sel].repeat_interleave(nc, 0) + off]))


def _uniform(dim, Dmax, D):
    s = 1 << D
    g = torch.arange(s, device="cuda", dtype=torch.int64)
    X = torch.stack(torch.meshgrid(*([g] * dim), indexing="ij"), -1).reshape(-1, dim) << (Dmax - D)
    return _Tree(dim, Dmax, torch.full((s ** dim,), D, device="cuda", dtype=torch.int64), X)


def _vortices(case, seed=None):
    """Vortex centres, strengths and core radii: separated places with seeded offsets and strengths
    (none: the ones whose tree the case has)."""
    r = np.random.default_rng(seed) if seed is not None else None
    L, k = case["L"], case["nvort"]
    at = {1: [(0.47, 0.53)], 2: [(0.24, 0.26), (0.77, 0.73)],
          4: [(0.24, 0.27), (0.76, 0.23), (0.26, 0.74), (0.73, 0.77)]}[k]

    def d(a):
        return a * (2 * r.random() - 1) if r else 0.0
    return np.array([[(x + d(0.004)) * L, (y + d(0.004)) * L, 5.0 + d(0.3), 1.0] for x, y in at])


def _vortex_tree(case, vort):
    """The tree a density-gradient criterion gives for the vortices: a leaf of level l is refined
    where its distance to a vortex axis is below the radius at which h |d rho/dr| = th_r; the radii
    of successive levels are kept far enough apart for 2:1 balance."""
    dim, L = case["dim"], case["L"]
    r = np.linspace(0.0, 0.5 * L, 20001)
    radii = []  # [level][vortex]
    for l in range(case["Dbase"], case["Dmax"]):
        row = []
        for v in vort:
            T = 1.0 - (GAMMA - 1) * v[2] ** 2 / (8 * GAMMA * np.pi ** 2) * np.exp(1 - (r / v[3]) ** 2)
            g = np.abs(np.gradient(T ** (1 / (GAMMA - 1)), r)) * L / 2 ** l
            hit = r[g > case["th_r"]]
            row.append(hit.max() if hit.size else 0.0)
        radii.append(row)
    for i in range(len(radii) - 2, -1, -1):
        gap = 1.5 * L / 2 ** (case["Dbase"] + i + 1)
        radii[i] = [max(a, b + gap) if b > 0 else a for a, b in zip(radii[i], radii[i + 1])]
    t = _uniform(dim, case["Dmax"], case["Dbase"])
    unit = L / (1 << case["Dmax"])
    for i, row in enumerate(radii):
        l = case["Dbase"] + i
        near = torch.zeros(t.M, dtype=torch.bool, device="cuda")
        for v, R in zip(vort, row):
            if R <= 0:
                continue
            d2 = torch.zeros(t.M, dtype=F64, device="cuda")
            for a in range(2):
                half = t.width(t.d).to(F64) * (unit / 2)
                c = t.X[:, a].to(F64) * unit + half - v[a]
                c = (c - L * torch.round(c / L)).abs()
                d2 += torch.clamp(c - half, min=0.0) ** 2
            near |= d2 < R * R
        sel = near & (t.d == l)
        t = _Tree(dim, case["Dmax"], *_children(t, sel))
    return t


def _points(t, L, o):
    """Physical x and y of every solution point, [M][N] each, and the element widths."""
    n, dim = o.n, t.dim
    unit = L / (1 << t.Dmax)
    h = t.width(t.d).to(F64) * unit
    pos = 0.5 * (o.xt + 1.0)
    i = torch.arange(n ** dim, device="cuda")
    x = t.X[:, :1].to(F64) * unit + h[:, None] * pos[i % n][None]
    y = t.X[:, 1:2].to(F64) * unit + h[:, None] * pos[(i // n) % n][None]
    return x, y, h


def _vortex_state(dim, L, vort, x, y, time):
    """Closed-form isentropic vortices advected at (1, 1): conserved variables [M][nv][N]."""
    du, dv, dT = torch.zeros_like(x), torch.zeros_like(x), torch.zeros_like(x)
    for xc, yc, beta, R in vort:
        dx, dy = x - (xc + time), y - (yc + time)
        dx = dx - L * torch.floor(dx / L + 0.5)
        dy = dy - L * torch.floor(dy / L + 0.5)
        r2 = (dx * dx + dy * dy) / (R * R)
        ex = torch.exp(0.5 * (1 - r2))
        du -= beta / (2 * math.pi) * dy / R * ex
        dv += beta / (2 * math.pi) * dx / R * ex
        dT -= (GAMMA - 1) * beta ** 2 / (8 * GAMMA * math.pi ** 2) * torch.exp(1 - r2)
    T = 1.0 + dT
    rho = T ** (1 / (GAMMA - 1))
    u, v = 1.0 + du, 1.0 + dv
    m = [rho * u, rho * v] + ([torch.zeros_like(x)] if dim == 3 else [])
    E = rho * T / (GAMMA - 1) + 0.5 * rho * (u * u + v * v)
    return torch.stack([rho] + m + [E], 1)


def _inputs(case, seed):
    """Vortices, tree (the same for every seed, as if adapted a few steps ago), initial state and
    time step of a cycle."""
    o = _Ops(case["p"])
    vort = _vortices(case, seed)
    t = _vortex_tree(case, _vortices(case))
    x, y, h = _points(t, case["L"], o)
    u = _vortex_state(case["dim"], case["L"], vort, x, y, 0.0)
    rho, m = u[:, 0], u[:, 1:-1]
    m2 = (m * m).sum(1)
    pr = (GAMMA - 1) * (u[:, -1] - 0.5 * m2 / rho)
    smax = float((torch.sqrt(m2) / rho + torch.sqrt(GAMMA * pr / rho)).max())
    hmin = case["L"] / (1 << case["Dmax"])
    dt = 0.3 * hmin / ((2 * case["p"] + 1) * smax)
    return o, vort, t, u, float("%.6g" % dt)


# ---- prepare / run ---------------------------------------------------------------------------------

STEPS = 10


def _mesh_config(case, vort, dt):
    return dict(dim=case["dim"], p=case["p"], L=case["L"], Dbase=case["Dbase"], Dmax=case["Dmax"], gamma=GAMMA,
                vort=vort, uinf=(1.0, 1.0, 0.0), rho_inf=1.0, p_inf=1.0, cfl=0.3, dt=dt, adapt_every=STEPS,
                indicator=0, th_refine=case["th_r"], th_coarsen=case["th_c"], precision=case["prec"], init_passes=0)


def _pinned(t):
    return torch.empty(t.shape, dtype=t.dtype, pin_memory=True).copy_(t)


def _room(case):
    """Leaves that the host buffers of a cycle have room for: the adaptation may grow the mesh."""
    return _leaf_count(case) * 3 // 2 + 256


def _torus(n, seed, dim, Dmin):
    """Points of a torus (2D: circle) in the unit box, moved periodically by whole cells of the coarsest
    level and reflected, both from the seed: another cloud with as many leaves."""
    r = np.random.default_rng(n)
    a, b = r.random(n) * 2 * np.pi, r.random(n) * 2 * np.pi
    if dim == 2:
        x = np.stack([0.5 + 0.3 * np.cos(a), 0.5 + 0.27 * np.sin(a)], 1)
    else:
        x = np.stack([0.5 + (0.28 + 0.1 * np.cos(b)) * np.cos(a), 0.5 + (0.26 + 0.1 * np.cos(b)) * np.sin(a),
                      0.5 + 0.1 * np.sin(b)], 1)
    x = (np.floor(x * 2.0 ** 30) + 0.5) / 2.0 ** 30  # so that the moves are exact
    for k in range(dim):
        x[:, k] = (x[:, k] + ((seed * (2 * k + 1)) % (1 << Dmin)) / (1 << Dmin)) % 1.0
        if (seed >> (Dmin + k)) & 1:
            x[:, k] = 1.0 - x[:, k]
    return x


def _learned_case(case):
    """The vortex mesh of the wanted size: depth from the element count, thresholds of the 3D runs."""
    dim, M = case["dim"], case["M"]
    Dbase = 3 if dim == 3 else 4
    Dmax = Dbase + 3
    while (1 << (dim * Dbase)) * 4 < M:
        Dbase += 1
        Dmax += 1
    return dict(dim=dim, p=case["p"], prec=0, L=20.0, Dbase=Dbase, Dmax=Dmax, nvort=1, th_r=0.05, th_c=0.0125)


def _params(n_in, seed):
    """Fan-in scaled uniform weights, zero biases, in the MLP's parameter layout."""
    r = np.random.default_rng(seed)
    out = []
    for fan, rows in ((n_in, 64), (64, 64), (64, 64), (64, 3)):
        out += [((r.random(fan * rows) * 2 - 1) * math.sqrt(6.0 / fan)), np.zeros(rows)]
    return torch.as_tensor(np.concatenate(out), dtype=torch.float32, device="cuda")


def _batch(case, seed):
    """Feature rows of two populations (quiet far field, vortex core) and labels that depend on them."""
    g = torch.Generator(device="cuda").manual_seed(seed)
    B, n_in = case["batch"], case["n_in"]
    s = torch.exp(torch.randn(B, 1, generator=g, device="cuda") * 1.5 - 1.0)
    X = torch.randn(B, n_in, generator=g, device="cuda") * s
    X[:, -1] = torch.randint(0, 4, (B,), generator=g, device="cuda") / 3.0
    y = ((s[:, 0] > 0.8).to(torch.int8) - (s[:, 0] < 0.2).to(torch.int8)).contiguous()
    return X.to(torch.bfloat16).contiguous(), y


CLASS_W = [1.5, 0.5, 2.0]


def prepare(case, seed):
    kind = case["kind"]
    if kind == "cycle":
        o, vort, t, u, dt = _inputs(case, seed)
        room = _room(case)
        return dict(kind=kind, mesh=fr.Mesh(_mesh_config(case, vort, dt)), keys=_pinned(t.key).numpy().view(np.uint64),
                    u=_pinned(u).numpy(),
                    keys_out=torch.zeros(room, dtype=torch.int64, pin_memory=True).numpy().view(np.uint64),
                    u_out=torch.zeros((room,) + u.shape[1:], dtype=F64, pin_memory=True).numpy())
    if kind == "tree":
        return dict(kind=kind, dim=case["dim"], Dmin=case["Dmin"], Dmax=case["Dmax"],
                    pts=torch.as_tensor(_torus(case["n"], seed, case["dim"], case["Dmin"]), device="cuda"))
    if kind == "learned":
        c = _learned_case(case)
        o, vort, t, u, dt = _inputs(c, seed)
        mesh = fr.Mesh(_mesh_config(c, vort, dt))
        mesh.set_state(t.key.cpu().numpy().view(np.uint64), u.cpu().numpy())
        return dict(kind=kind, mesh=mesh, params=_params(55 if c["dim"] == 3 else 19, seed))
    X, y = _batch(case, seed)
    P = _params(case["n_in"], seed)
    return dict(kind=kind, X=X, y=y, P=P, m=torch.zeros_like(P), v=torch.zeros_like(P), step=0,
                loss=torch.zeros(1, dtype=torch.float32, device="cuda"))


def run(state):
    s = state
    kind = s["kind"]
    if kind == "cycle":
        m = s["mesh"]
        m.set_state(s["keys"], s["u"])
        m.set_time(0.0)
        m.run(STEPS)
        n = m.norms()
        m.leaves(out=s["keys_out"])
        m.state(out=s["u_out"])
        return dict(leaves=n["M"], keys=s["keys_out"].view(np.int64), state=s["u_out"],
                    norms=np.array([n["l2_rho"], n["min_rho"], n["min_p"]] + n["integral"]))
    if kind == "tree":
        keys = fr.tree_complete(s["dim"], s["Dmin"], s["Dmax"], 1.0, s["pts"])
        return dict(complete=keys.view(np.int64), balanced=fr.tree_balance(s["dim"], s["Dmax"], keys).view(np.int64))
    if kind == "learned":
        X = s["mesh"].features()
        logits, flags = fr.mlp_forward(s["params"], X)
        return dict(features=X, logits=logits, flags=flags)
    fr.mlp_train_step(s["P"], s["m"], s["v"], s["step"], s["X"], s["y"], CLASS_W, 2e-3, s["loss"])
    s["step"] += 1
    return dict(params=s["P"], m=s["m"], v=s["v"], loss=s["loss"])


# ---- what a pass cannot do without -----------------------------------------------------------------

_SIZE = {}


def _leaf_count(case):
    """Leaves of the vortex tree of this case."""
    key = tuple(sorted((k, v) for k, v in case.items() if k != "name"))
    if key not in _SIZE:
        _SIZE[key] = _vortex_tree(case, _vortices(case)).M
    return _SIZE[key]


def work(case):
    kind = case["kind"]
    if kind == "cycle":
        d, n = case["dim"], case["p"] + 1
        M, N, nv, NF = _leaf_count(case), n ** d, d + 2, n ** (d - 1)
        # per point and stage: pointwise flux, folded derivative with correction, RK combination and
        # traces; per conforming face point the Rusanov flux (d faces per element)
        point = 3 * d + 4 + d * (d + 3) + d * nv * (2 * n + 3) + 6 * nv + 4 * d * nv
        face = 2 * (3 * d + 15) + 3 + 4 * nv
        stages = 3 * STEPS
        # each stage reads its state and the step's first one and writes the new one; the faces'
        # traces and common fluxes are exchanged between elements once, in the form's storage type
        exch = 4 * d * nv * NF * (4 if case["prec"] == 1 else 8) * 2
        b = stages * M * (3 * nv * N * 8 + exch) + 2 * M * (nv * N + 1) * 8
        return {"bytes": b, "flops": stages * M * (N * point + d * NF * face)}
    if kind == "tree":
        # points in; at most one cell of the finest level per point and its seven siblings out, twice
        return {"bytes": case["n"] * case["dim"] * 8 + 2 * 8 * 2 * case["n"], "flops": 60 * case["n"]}
    if kind == "learned":
        c = _learned_case(case)
        d, n = c["dim"], c["p"] + 1
        M, N, nv, IN = _leaf_count(c), n ** d, d + 2, 2 * 3 ** d + 1
        interp = sum(2 * n * 3 ** (k + 1) * n ** (d - 1 - k) for k in range(d))
        mlp = 2 * (IN * 64 + 2 * 64 * 64 + 3 * 64)
        return {"bytes": M * (nv * N * 8 + 8 + 4 * IN + 13), "flops": M * (nv * interp + mlp)}
    B, IN = case["batch"], case["n_in"]
    macs = IN * 64 + 2 * 64 * 64 + 3 * 64
    npar = IN * 64 + 64 + 2 * (64 * 64 + 64) + 3 * 64 + 3
    return {"bytes": B * (2 * IN + 1) + 6 * 4 * npar, "flops": 6 * macs * B}


# ---- the method in plain FP64 ------------------------------------------------------------------------

def _grid(u, o, dim):
    return u.reshape(u.shape[0], u.shape[1], *([o.n] * dim))  # [.., (z,) y, x]


def _contract(u, A, dim, axis):
    """A [r, n] along `axis` (x last in memory) of [M, nv, (z,) y, x]."""
    return torch.movedim(torch.tensordot(torch.movedim(u, -1 - axis, -1), A, ([-1], [1])), -1, -1 - axis)


def _flux(u, axis, dim):
    rho, E = u[:, 0], u[:, -1]
    m = u[:, 1:-1]
    pr = (GAMMA - 1) * (E - 0.5 * (m * m).sum(1) / rho)
    v = m[:, axis] / rho
    f = u * v[:, None]
    f[:, 1 + axis] += pr
    f[:, -1] += pr * v
    return f, pr, v


def _rusanov(qL, qR, axis, dim):
    fL, pL, vL = _flux(qL, axis, dim)
    fR, pR, vR = _flux(qR, axis, dim)
    lam = torch.maximum(vL.abs() + torch.sqrt(GAMMA * pL / qL[:, 0]), vR.abs() + torch.sqrt(GAMMA * pR / qR[:, 0]))
    return 0.5 * (fL + fR) - 0.5 * lam[:, None] * (qR - qL)


def _faces(t):
    """Per axis: conforming pairs (minus, plus) and, per side, hanging (fine, coarse, slot bits)."""
    out = []
    w, full = t.width(t.d), 1 << t.Dmax
    for a in range(t.dim):
        row = []
        for side in (0, 1):
            X = t.X.clone()
            X[:, a] = (X[:, a] + (w if side else -w)) % full
            j = t.locate(X)
            same, coarse = t.d[j] == t.d, t.d[j] < t.d
            conf = torch.nonzero(same)[:, 0]
            fine = torch.nonzero(coarse)[:, 0]
            bits = [(t.X[fine, b] // w[fine]) % 2 for b in range(t.dim) if b != a]
            row.append((conf, j[conf], fine, j[fine], bits))
        out.append(row)
    return out


def _rhs(u, t, faces, o, L):
    dim, n = t.dim, o.n
    g = _grid(u, o, dim)
    h = t.width(t.d).to(F64) * (L / (1 << t.Dmax))
    shape = [t.M] + [1] * (dim + 1)
    R = torch.zeros_like(g)
    inner = dim - 1
    for a in range(dim):
        tr = [_contract(g, l[None], dim, a).squeeze(-1 - a).reshape(t.M, dim + 2, -1) for l in (o.lm, o.lp)]
        F = [torch.zeros_like(tr[0]), torch.zeros_like(tr[0])]
        e, nb = faces[a][1][0], faces[a][1][1]
        f = _rusanov(tr[1][e], tr[0][nb], a, dim)
        F[1][e] = f
        F[0][nb] = f
        for side in (0, 1):
            _, _, fine, coarse, bits = faces[a][side]
            if not fine.numel():
                continue
            slot = bits[0] if inner == 1 else bits[0] + 2 * bits[1]
            for s in range(1 << inner):
                k = torch.nonzero(slot == s)[:, 0]
                if not k.numel():
                    continue
                fe, ce, hs = fine[k], coarse[k], [(s >> b) & 1 for b in range(inner)]
                c = tr[1 - side][ce].reshape(-1, dim + 2, *([n] * inner))
                for b in range(inner):
                    c = _contract(c, o.I[hs[b]], inner, b)
                c = c.reshape(-1, dim + 2, n ** inner)
                q = tr[side][fe]
                f = _rusanov(q, c, a, dim) if side else _rusanov(c, q, a, dim)
                F[side][fe] = f
                b_ = f.reshape(-1, dim + 2, *([n] * inner))
                for b in range(inner):
                    b_ = _contract(b_, o.P[hs[b]], inner, b)
                F[1 - side].index_add_(0, ce, b_.reshape(-1, dim + 2, n ** inner))
        fx = _flux(g, a, dim)[0]
        d = _contract(fx, o.D, dim, a)
        for gs, l, Fs in ((o.gL, o.lm, F[0]), (o.gR, o.lp, F[1])):
            jump = Fs.reshape(t.M, dim + 2, *([n] * inner)).unsqueeze(-1 - a) - _contract(fx, l[None], dim, a)
            d = d + jump * gs.reshape([n] + [1] * a)
        R = R - d * (2.0 / h).reshape(shape)
    return R.reshape(u.shape)


def _flags(u, t, o, case):
    g = _grid(u[:, :1], o, t.dim)
    g2 = sum(_contract(g, o.D, t.dim, a) ** 2 for a in range(t.dim))
    eta = 2 * torch.sqrt(g2.reshape(t.M, -1).amax(1))
    return (eta > case["th_r"]).to(torch.int64) - (eta < case["th_c"]).to(torch.int64)


def _edit(t, flags, case):
    refine = (flags > 0) & (t.d < t.Dmax)
    w = t.width(t.d)
    span = 2 * w
    parent = t.X // span[:, None] * span[:, None]
    pkey = (_interleave(parent, t.dim) << t.mb) | (t.d - 1)
    ok = (flags < 0) & (t.d > case["Dbase"])
    uniq, inv, cnt = torch.unique(torch.where(ok, pkey, -1 - torch.arange(t.M, device="cuda")), return_inverse=True,
                                  return_counts=True)
    fuse = ok & (cnt[inv] == (1 << t.dim))
    head = fuse & (parent == t.X).all(1)
    keep = ~refine & ~fuse
    cd, cX = _children(t, refine)
    rest = torch.cat([keep[~refine], torch.ones(cd.numel() - int((~refine).sum()), dtype=torch.bool, device="cuda")])
    return _Tree(t.dim, t.Dmax, torch.cat([cd[rest], t.d[head] - 1]), torch.cat([cX[rest], parent[head]]))


def _balance(t, Dlow):
    offs = torch.tensor([[(k // 3 ** a) % 3 - 1 for a in range(t.dim)] for k in range(3 ** t.dim)], device="cuda")
    full = 1 << t.Dmax
    for D in range(t.Dmax, max(Dlow, 2) - 1, -1):
        while True:
            X = t.X[t.d == D]
            split = torch.zeros(t.M, dtype=torch.bool, device="cuda")
            for k in range(3 ** t.dim):
                j = t.locate((X + offs[k] * (full >> D)) % full)
                split[j[t.d[j] < D - 1]] = True
            if not bool(split.any()):
                break
            t = _Tree(t.dim, t.Dmax, *_children(t, split))
    return t


def _transfer(u, a, b, o):
    """State u of tree a on tree b: copy, interpolation of the ancestor, projection of the children."""
    dim, n, nc = a.dim, o.n, 1 << a.dim
    j = a.locate(b.X)
    first = torch.searchsorted(a.key, b.key)
    out = torch.empty(b.M, u.shape[1], u.shape[2], dtype=F64, device="cuda")
    same = a.d[j] == b.d
    out[same] = u[j[same]]
    inside = torch.nonzero(a.d[j] < b.d)[:, 0]
    if inside.numel():
        A = j[inside]
        wa, wb = a.width(a.d[A]).to(F64), b.width(b.d[inside]).to(F64)
        g = _grid(u[A], o, dim)
        for ax in range(dim):
            xi = -1 + 2 * ((b.X[inside, ax] - a.X[A, ax]).to(F64)[:, None] + 0.5 * (o.xt + 1) * wb[:, None]) / wa[:, None]
            W = torch.ones(inside.numel(), n, n, dtype=F64, device="cuda")
            for m in range(n):
                for k in range(n):
                    if k != m:
                        W[:, :, m] *= (xi - o.xt[k]) / (o.xt[m] - o.xt[k])
            g = torch.movedim(g, -1 - ax, -1)
            sh = g.shape
            g = torch.bmm(g.reshape(sh[0], -1, n), W.transpose(1, 2)).reshape(sh)
            g = torch.movedim(g, -1, -1 - ax)
        out[inside] = g.reshape(inside.numel(), u.shape[1], -1)
    fused = torch.nonzero(a.d[j] > b.d)[:, 0]
    if fused.numel():
        acc = 0
        for c in range(nc):
            g = _grid(u[first[fused] + c], o, dim)
            for ax in range(dim):
                g = _contract(g, o.P[(c >> ax) & 1], dim, ax)
            acc = acc + g
        out[fused] = acc.reshape(fused.numel(), u.shape[1], -1)
    return out


def _norms(u, t, o, case, vort, time):
    dim, n = t.dim, o.n
    x, y, h = _points(t, case["L"], o)
    ex = _vortex_state(dim, case["L"], vort, x, y, time)
    i = torch.arange(n ** dim, device="cuda")
    W = o.wt[i % n] * o.wt[(i // n) % n] * (o.wt[i // (n * n)] if dim == 3 else 1.0)
    WJ = W[None] * ((0.5 * h) ** dim)[:, None]
    pr = (GAMMA - 1) * (u[:, -1] - 0.5 * (u[:, 1:-1] ** 2).sum(1) / u[:, 0])
    return torch.cat([torch.stack([torch.sqrt((WJ * (ex[:, 0] - u[:, 0]) ** 2).sum()), u[:, 0].min(), pr.min()]),
                      (u * WJ[:, None]).sum((0, 2))])


def _layers(P, n_in):
    out, k = [], 0
    for fan, rows in ((n_in, 64), (64, 64), (64, 64), (64, 3)):
        out.append((P[k:k + fan * rows].reshape(rows, fan), P[k + fan * rows:k + fan * rows + rows]))
        k += fan * rows + rows
    return out


def _mlp(P, X, n_in):
    z = X
    for k, (W, b) in enumerate(_layers(P, n_in)):
        z = z @ W.T + b
        if k < 3:
            z = 0.5 * z * (1 + torch.erf(z / math.sqrt(2.0)))
    return z


def exact(case, seed):
    kind = case["kind"]
    if kind == "tree":
        return None  # whole numbers only
    if kind == "cycle":
        o, vort, t, u, dt = _inputs(case, seed)
        faces = _faces(t)
        for _ in range(STEPS):
            u1 = u + dt * _rhs(u, t, faces, o, case["L"])
            u2 = 0.75 * u + 0.25 * (u1 + dt * _rhs(u1, t, faces, o, case["L"]))
            u = (u + 2.0 * (u2 + dt * _rhs(u2, t, faces, o, case["L"]))) / 3.0
        b = _balance(_edit(t, _flags(u, t, o, case), case), case["Dbase"] + 2)
        u = _transfer(u, t, b, o)
        out = torch.zeros((_room(case),) + u.shape[1:], dtype=F64, device="cuda")
        out[:b.M] = u
        return dict(leaves=None, keys=None, state=out, norms=_norms(u, b, o, case, vort, STEPS * dt))
    if kind == "learned":
        c = _learned_case(case)
        o, vort, t, u, dt = _inputs(c, seed)
        g = _grid(u, o, t.dim)
        A = torch.as_tensor(_lagrange(o.x, np.polynomial.legendre.leggauss(3)[0]), dtype=F64, device="cuda")
        for a in range(t.dim):
            g = _contract(g, A, t.dim, a)
        g = g.reshape(t.M, t.dim + 2, -1)
        rho = g[:, 0]
        pr = (GAMMA - 1) * (g[:, -1] - 0.5 * (g[:, 1:-1] ** 2).sum(1) / rho)
        dev = [100 * (q - q.mean(1, keepdim=True)) / q.mean(1, keepdim=True) for q in (rho, pr)]
        level = (t.d - c["Dbase"]).to(F64)[:, None] / max(1, c["Dmax"] - c["Dbase"])
        X = torch.cat(dev + [level], 1)
        n_in = X.shape[1]
        return dict(features=X, logits=_mlp(_params(n_in, seed).to(F64), X, n_in), flags=None)
    X, y = _batch(case, seed)
    P = _params(case["n_in"], seed).to(F64).requires_grad_(True)
    logp = torch.log_softmax(_mlp(P, X.to(F64), case["n_in"]), 1)
    cls = (y + 1).to(torch.int64)
    w = torch.tensor(CLASS_W, dtype=F64, device="cuda")[cls]
    loss = -(w * logp.gather(1, cls[:, None])[:, 0]).sum() / w.sum()
    g, = torch.autograd.grad(loss, P)
    with torch.no_grad():
        m, v = 0.1 * g, 0.001 * g * g
        new = P - 2e-3 * (m / 0.1) / (torch.sqrt(v / 0.001) + 1e-8)
    return dict(params=new.detach(), m=m, v=v, loss=loss.detach().reshape(1))
