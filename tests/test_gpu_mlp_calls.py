"""The training calls' contract: the loss's factor given or formed, refusals that write nothing, and the Adam
update against its formula in FP64 on the gradient that mlp_grad returns."""
import ctypes as C

import numpy as np
import pytest

from paper_2306_06744_gb300 import fr
from paper_2306_06744_gb300 import workloads as W

pytestmark = pytest.mark.gpu

N_IN = 19


def _case(B, seed):
    import torch
    P = ((W.random_uniform(fr.mlp_param_count(N_IN), seed) - 0.5) * 0.5).astype(np.float32)
    X = torch.tensor((W.random_uniform(B * N_IN, seed + 1).reshape(B, N_IN) - 0.5) * 6, dtype=torch.float32)
    y = (np.floor(W.random_uniform(B, seed + 2) * 3) - 1).astype(np.int8)
    return torch.from_numpy(P).cuda(), X.to(torch.bfloat16).cuda(), torch.from_numpy(y).cuda()


def _raw_grad(P, X, y, cw, alloc=False):
    import torch
    g, loss = torch.full_like(P, 7.0), torch.full((1,), 7.0, device="cuda")
    w = np.array(cw, dtype=np.float32)
    p = [C.c_void_p(t.data_ptr()) for t in (P, X, y, g, loss)]
    args = [N_IN, p[0], p[1], p[2], X.shape[0], C.c_void_p(w.ctypes.data), p[3], p[4], None]
    lib = fr.load()
    torch.cuda.synchronize()
    rc = lib.fr_mlp_grad_alloc(*args, None) if alloc else lib.fr_mlp_grad(*args)
    return rc, g.cpu().numpy(), float(loss.item())


@pytest.mark.parametrize("B", [1, 127, 129, 4096])
def test_factor_given_or_formed(B):
    P, X, y = _case(B, 11)
    w = np.array([1.5, 0.5, 2.0], dtype=np.float32)
    total = w.astype(np.float64)[y.cpu().numpy().astype(int) + 1].sum()
    rc, g, loss = _raw_grad(P, X, y, [*w, np.float32(1.0 / total)])
    assert rc == 0 and loss > 0.0 and np.abs(g).max() > 0.0
    rc2, g2, loss2 = _raw_grad(P, X, y, [*w, 0.0], alloc=True)
    assert rc2 == 0 and np.array_equal(g, g2) and loss == loss2
    lw, gw = fr.mlp_grad(P, X, y, w)
    assert lw == loss and np.array_equal(gw.cpu().numpy(), g)
    # the plain form takes a factor of zero as it is
    rc3, g3, loss3 = _raw_grad(P, X, y, [*w, 0.0])
    assert rc3 == 0 and loss3 == 0.0 and not g3.any()


@pytest.mark.parametrize("label", [2, -2, 127, -128])
def test_labels_out_of_range_write_nothing(label):
    import torch
    P, X, y = _case(300, 21)
    m, v = torch.rand_like(P), torch.rand_like(P)
    loss = torch.full((1,), 7.0, device="cuda")
    y[137] = label
    was = [t.clone() for t in (P, m, v, loss)]
    with pytest.raises(fr.FRError) as e:
        fr.mlp_train_step(P, m, v, 3, X, y, [1.0, 1.0, 1.0], 1e-3, loss)
    assert e.value.code == fr.FR_EINVAL
    assert all(torch.equal(a, b) for a, b in zip(was, (P, m, v, loss)))
    for alloc, f in ((False, 0.01), (True, 0.0)):
        rc, g, lo = _raw_grad(P, X, y, [1.0, 1.0, 1.0, f], alloc)
        assert rc == fr.FR_EINVAL and (g == 7.0).all() and lo == 7.0


@pytest.mark.parametrize("w_keep", [0.0, 1e-42])  # 1 / (300 * 1e-42) is past the FP32 range
def test_weights_without_a_finite_factor_write_nothing(w_keep):
    import torch
    P, X, y = _case(300, 31)
    y.zero_()  # only class 0 is present
    m, v = torch.rand_like(P), torch.rand_like(P)
    was = [t.clone() for t in (P, m, v)]
    with pytest.raises(fr.FRError) as e:
        fr.mlp_train_step(P, m, v, 0, X, y, [1.0, w_keep, 1.0], 1e-3)
    assert e.value.code == fr.FR_EINVAL
    with pytest.raises(fr.FRError):
        fr.mlp_grad(P, X, y, [1.0, w_keep, 1.0])
    assert all(torch.equal(a, b) for a, b in zip(was, (P, m, v)))


@pytest.mark.parametrize("B", [64, 3000])
def test_adam_update_is_its_formula(B):
    import torch
    P, X, y = _case(B, 41)
    m, v = torch.zeros_like(P), torch.zeros_like(P)
    lr, b1, b2, eps, u = 2e-3, float(np.float32(0.9)), float(np.float32(0.999)), 1e-8, 2.0 ** -24
    cw = [1.5, 0.5, 2.0]
    for step in range(3):
        _, g = fr.mlp_grad(P, X, y, cw)
        p0, m0, v0, g = (t.double().cpu().numpy() for t in (P, m, v, g))
        fr.mlp_train_step(P, m, v, step, X, y, cw, lr)
        want_m = b1 * m0 + (1 - b1) * g
        want_v = b2 * v0 + (1 - b2) * g * g
        got_p, got_m, got_v = (t.double().cpu().numpy() for t in (P, m, v))
        # three (four) roundings of the terms
        assert (np.abs(got_m - want_m) <= 3 * u * (np.abs(b1 * m0) + np.abs((1 - b1) * g)) + 1e-44).all()
        assert (np.abs(got_v - want_v) <= 4 * u * want_v + 1e-44).all()
        # the step from the moments just checked: its own eight roundings, and those of the powers in
        # 1 - b^(step + 1), 4 u beside 1 - b2^(step + 1) (half of it through the root)
        c1, c2 = 1 - b1 ** (step + 1), 1 - b2 ** (step + 1)
        d = lr * (got_m / c1) / (np.sqrt(got_v / c2) + eps)
        assert (np.abs(got_p - (p0 - d)) <= (8 + 4 / c1 + 2 / c2) * u * np.abs(d) + u * np.abs(p0)).all()
