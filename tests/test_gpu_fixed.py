"""The FP64 form's fixed-point contractions and its square root and reciprocal on the GPU."""
import os
import subprocess
import tempfile

import numpy as np
import pytest

import oracle as O
from paper_2306_06744_gb300 import fr
from paper_2306_06744_gb300 import workloads as W
from tests.test_gpu_fr import _random_tree, _smooth_state, rel_l2

pytestmark = pytest.mark.gpu

HERE = os.path.dirname(os.path.abspath(__file__))
CSRC = os.path.join(os.path.dirname(HERE), "paper_2306_06744_gb300", "csrc")


def test_root_and_reciprocal_against_correct_rounding():
    # sqrt_t: Markstein's correction leaves half an ulp and 2^-66, so at most 1 ulp from the correctly
    # rounded root; rcp_t: e^3 = 2^-69 plus the rounding of its last multiply-add, at most 1 ulp
    from paper_2306_06744_gb300 import build as B
    exe = os.path.join(tempfile.mkdtemp(), "root_check")
    cmd = [B._nvcc(), *B.ARCH, "-O3", "-std=c++17", "-I" + CSRC, os.path.join(HERE, "cuda", "root_check.cu"), "-o", exe]
    subprocess.run(cmd, check=True, capture_output=True, text=True)
    out = subprocess.run([exe], check=True, capture_output=True, text=True, timeout=120).stdout
    vals = {k: int(v) for k, v in (line.split() for line in out.strip().splitlines())}
    assert vals["sqrt"] <= 1 and vals["rcp"] <= 1 and vals["special"] == 0, vals


@pytest.mark.parametrize("dim,p,Dbase,Dmax,seed", [(2, 1, 2, 6, 11), (2, 2, 2, 6, 12), (2, 3, 2, 6, 13), (2, 4, 2, 5, 14),
                                                   (3, 1, 1, 4, 15), (3, 2, 1, 4, 16), (3, 3, 1, 3, 17), (3, 4, 1, 3, 18)])
def test_rhs_far_from_unit_scale(dim, p, Dbase, Dmax, seed):
    # Group exponents: density 2^-40, momenta and energy in units 2^20 faster and 2^40 more energetic
    # (the equations are homogeneous: powers of two scale every value exactly, so the residual in
    # these units holds the same relative bar as in unit scale)
    cfg = dict(W.config("vortex2d_p2_small" if dim == 2 else "vortex3d_p2_tube"), dim=dim, p=p, Dbase=Dbase, Dmax=Dmax,
               init_passes=0, indicator=2, dt=1e-3)
    keys = _random_tree(dim, Dbase, Dmax, seed)
    u = _smooth_state(cfg, keys, seed)
    s = np.array([2.0 ** -40] + [2.0 ** -20] * dim + [1.0])[None, :, None]
    g, o = fr.Mesh(cfg), O.OracleMesh(cfg)
    o.set_state(keys, u)
    g.set_state(keys, u * s)
    R = g.rhs() / (s * 2.0 ** 20)  # time runs 2^20 faster
    want = o.rhs()
    for v in range(dim + 2):
        assert rel_l2(R[:, v], want[:, v]) < 1e-12, v


def test_nan_in_one_element_reaches_its_residual():
    cfg = dict(W.config("vortex2d_p2_small"), init_passes=0, indicator=2, dt=1e-3)
    keys = _random_tree(2, cfg["Dbase"], cfg["Dmax"], 5)
    u = _smooth_state(cfg, keys, 5)
    u[7, 0, 4] = np.nan
    g = fr.Mesh(cfg)
    g.set_state(keys, u)
    R = g.rhs()
    assert np.isnan(R[7, 0]).any() and not np.isnan(R).all()
