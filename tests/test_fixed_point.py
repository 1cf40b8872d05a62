"""The fixed-point arithmetic of the FP64 form's quadrature points
(bem_fixed.cuh), on the host against long double (tests/fixed_point_check.cpp,
built here with the host compiler).

Bounds: the squared length drops three products of signed low words, at most
2^62 / 2^64 each, and rounds once: below 1.5 units.  The reciprocal square root
carries a float correction of a term below 2^-31 (2^-55) and truncations of
2^-58: below 2^-53, as a rounded double.  The sine and cosine truncate a tail of
2^-45 units times z^4 <= 2^-8: below 2^-52.  Distances below a sixteenth of the
scale are flagged."""
import os
import shutil
import subprocess

import pytest

ROOT = os.path.dirname(os.path.dirname(os.path.abspath(__file__)))


def test_fixed_point_arithmetic(tmp_path):
    cxx = shutil.which("g++") or shutil.which("c++")
    inc = "/usr/local/cuda/include"
    if cxx is None or not os.path.exists(os.path.join(inc, "cuda_runtime.h")):
        pytest.skip("no host C++ compiler or CUDA headers")
    exe = str(tmp_path / "fixed_point_check")
    subprocess.run([cxx, "-O2", "-std=c++17", "-I", inc, "-I",
                    os.path.join(ROOT, "paper_1510_07244_gb300", "csrc"), "-x", "c++",
                    os.path.join(ROOT, "tests", "fixed_point_check.cpp"), "-o", exe], check=True)
    out = subprocess.run([exe], capture_output=True, text=True, check=True).stdout
    got = {line.split()[0]: [float(v) for v in line.split()[1:]] for line in out.splitlines()}
    assert got["norm2"][0] < 1.5
    for kb in range(5):
        worst, flagged = got[f"rinv{kb}"]
        assert worst < 2.0 ** -53 and flagged < 40, (kb, worst, flagged)   # flags: rounding at the edge
    assert got["flags"] == [4.0]
    assert got["sincos"][0] < 2.0 ** -52
