"""CPU check of the scaling of face cotangents (cot_exponent, ff_of_shifted and shifted in adjoint_ff.cuh),
compiled for the host by nvcc: zeros stay exact zeros, alone and beside components of any size, and a
cotangent whose size leaves no room for the two floats or for the way back is left to FP64.  Bound: a
scaled component is its FP64 value times a power of two to 2^-47 of itself."""
import math
import os
import shutil
import subprocess

import pytest

from conftest import ROOT


@pytest.fixture(scope="module")
def check(tmp_path_factory):
    nvcc = shutil.which("nvcc") or "/usr/local/cuda/bin/nvcc"
    if not os.path.exists(nvcc):
        pytest.skip("nvcc not available")
    exe = tmp_path_factory.mktemp("cot") / "check_cotangent_scaling"
    src = os.path.join(ROOT, "tests", "native", "check_cotangent_scaling.cu")
    r = subprocess.run([nvcc, "-std=c++17", "-O2", "-Xcompiler", "-ffp-contract=off", "-diag-suppress", "177", src,
                        "-o", str(exe)], capture_output=True, text=True)
    assert r.returncode == 0, r.stderr

    def run(x):
        out = subprocess.run([str(exe)], input=" ".join(float(v).hex() for v in x) + "\n", capture_output=True,
                             text=True, check=True).stdout.split()
        return int(out[0]), [float(v) for v in out[1:6]], int(out[6]), float(out[7])
    return run


def test_zero_cotangents_give_zero(check):
    for x in ([0.0] * 5, [-0.0] * 5):
        taken, g, _, slot = check(x)
        assert taken == 1 and g == [0.0] * 5 and slot == 0.0


@pytest.mark.parametrize("e", [-1070, -1022, -1000, -950, -900, -500, -1, 0, 1, 500, 870, 950, 1023])
def test_components_keep_their_value_or_go_to_fp64(check, e):
    x = [math.ldexp(1.3, e), 0.0, math.ldexp(-0.7, e - 20), 0.0, math.ldexp(0.9, e - 3)]
    taken, g, k, _ = check(x)
    assert taken == (-912 < e < 880)
    if taken:
        for a, b in zip(x, g):
            assert abs(b - math.ldexp(a, -k)) <= 2.0 ** -47 * abs(math.ldexp(a, -k))
