"""The block fixed point of the FP64 form's contractions (fr_fixed.cuh), run on the host: every result
within the bound that its operand splitting implies, for the term counts of all degrees and dimensions
(2 to 5 for traces, 8 to 21 for the derivative with its corrections) and the interface kernel's sums of
products, over group exponents from 2^-900
to 2^900 and spreads to 2^80 within a group (tests/cuda/fixed_check.cu)."""
import os
import subprocess
import tempfile

HERE = os.path.dirname(os.path.abspath(__file__))
CSRC = os.path.join(os.path.dirname(HERE), "paper_2306_06744_gb300", "csrc")
TERMS = [2, 3, 4, 5, 8, 10, 12, 14, 15, 18, 21]


def test_fixed_point_contraction_bounds():
    from paper_2306_06744_gb300 import build as B
    exe = os.path.join(tempfile.mkdtemp(), "fixed_check")
    cmd = [B._nvcc(), *B.ARCH, "-O2", "-std=c++17", "-I" + CSRC, os.path.join(HERE, "cuda", "fixed_check.cu"), "-o", exe]
    subprocess.run(cmd, check=True, capture_output=True, text=True)
    out = subprocess.run([exe, *map(str, TERMS)], check=True, capture_output=True, text=True, timeout=120).stdout
    vals = dict(line.split() for line in out.strip().splitlines())
    for n in TERMS:
        assert 0.0 < float(vals["n%d" % n]) <= 1.0, vals
    assert 0.0 < float(vals["dot"]) <= 1.0 and 0.0 < float(vals["squares"]) <= 1.0, vals
    assert float(vals["double"]) <= 1.0 and float(vals["zero"]) == 0.0 and vals["nan"] == "1", vals
