"""The FP64 form's interface flux (rusanov2_fx) on the host against the same flux in long double, with the
states that its integer products could get wrong: units in which all values are tiny (from 2^-470) or huge, one
side up to 1e8 times as dense, one side's pressure negative (its wave speed is not a number, and its speed may
exceed the other side's wave speed), NaN of either sign and infinities (tests/cuda/flux_check.cu, which
derives the bounds)."""
import os
import subprocess
import tempfile

import pytest

HERE = os.path.dirname(os.path.abspath(__file__))
ROOT = os.path.dirname(HERE)


@pytest.fixture(scope="module")
def results():
    from paper_2306_06744_gb300 import build as B
    exe = os.path.join(tempfile.mkdtemp(), "flux_check")
    cmd = [B._nvcc(), *B.ARCH, "-O2", "-std=c++17", "-I" + os.path.join(ROOT, "paper_2306_06744_gb300", "csrc"),
           "-I" + os.path.join(ROOT, "include"), os.path.join(HERE, "cuda", "flux_check.cu"), "-o", exe]
    subprocess.run(cmd, check=True, capture_output=True, text=True)
    out = subprocess.run([exe], check=True, capture_output=True, text=True, timeout=120).stdout
    return dict(line.split() for line in out.strip().splitlines())


@pytest.mark.parametrize("dim", [2, 3])
@pytest.mark.parametrize("kind", ["plain", "smallest", "tiny", "huge", "jump", "negative_pressure"])
def test_flux_within_its_bound(results, kind, dim):
    assert 0.0 < float(results["%s%d" % (kind, dim)]) <= 1.0, results


def test_special_values_are_not_lost(results):
    assert results["special2"] == results["special3"] == results["larger"] == "0", results
