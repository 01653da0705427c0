"""CPU check of the two-float terms of the FP64 face kernels (ff_math.cuh, face_ff.cuh), compiled for
the host by nvcc: on seeded windows and face states inside the limits of the two-float path, the
reconstructed values and the HLLC flux formed with them are as near to the same formulas in long
double as the FP64 formulas are.  Bounds: a split FP64 number keeps 2^-48 of itself and comes back
within 2^-52; the root-mean-square errors over 20,000 samples are at most those of the FP64 formulas
plus 3 % (the statistical spread of the two means, 2 / sqrt(20000), doubled).  TENO6-A's decisions in
FP32 are the FP64 ones wherever their error bound calls them clear, which is all but 1e-3 of them."""
import os
import shutil
import subprocess

import pytest

from conftest import ROOT


def test_two_float_terms_are_as_exact_as_fp64(tmp_path):
    nvcc = shutil.which("nvcc") or "/usr/local/cuda/bin/nvcc"
    if not os.path.exists(nvcc):
        pytest.skip("nvcc not available")
    exe = tmp_path / "check_face_ff"
    src = os.path.join(ROOT, "tests", "native", "check_face_ff.cu")
    # the error-free sums must not be contracted by the host compiler
    r = subprocess.run([nvcc, "-std=c++17", "-O2", "-Xcompiler", "-ffp-contract=off", "-diag-suppress", "177",
                        src, "-o", str(exe)], capture_output=True, text=True)
    assert r.returncode == 0, r.stderr
    out = subprocess.run([str(exe)], capture_output=True, text=True).stdout.split("\n")
    rows = {p[0]: (float(p[1]), float(p[2])) for p in (line.split() for line in out) if p}
    assert len(rows) == 1 + 6 + 27 + 4
    split, back = rows.pop("split")
    assert split <= 2.0 ** -48 and back <= 2.0 ** -52
    for kind in range(4):                      # smooth, noise, steps, near zero
        left_open, wrong = rows.pop("teno%d" % kind)
        assert wrong == 0.0 and left_open < 1e-3
    for name, (fp64, ff) in rows.items():
        assert ff <= 1.03 * fp64, (name, fp64, ff)
