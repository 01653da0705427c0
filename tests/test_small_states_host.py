"""CPU check of the two-float WENO5 weights where cell differences are near their epsilon, compiled for the host
by nvcc.  At the smallest states of the two-float path (1.9e-6) the face values are as near to the
definition in long double as the FP64 formula's, within the 3 % of two means over 20,000 samples.  For a
field about zero (a velocity) they keep 2^-40 of its amplitude (two floats to 2^-47, times a condition of
the weights' quotients of up to 100) and 2^-94 (a correction below 2^-70 is converted with 24 bits)."""
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
    exe = tmp_path_factory.mktemp("small") / "check_small_states"
    src = os.path.join(ROOT, "tests", "native", "check_small_states.cu")
    r = subprocess.run([nvcc, "-std=c++17", "-O2", "-Xcompiler", "-ffp-contract=off", "-diag-suppress", "177", src,
                        "-o", str(exe)], capture_output=True, text=True)
    assert r.returncode == 0, r.stderr

    def run(base, amp, eps):
        out = subprocess.run([str(exe)] + [repr(v) for v in (base, amp, eps)], capture_output=True, text=True, check=True)
        rows = [[float(v) for v in line.split()] for line in out.stdout.splitlines()]
        assert len(rows) == 2 and all(r[0] == 20000 for r in rows)
        return rows
    return run


@pytest.mark.parametrize("amp", [1e-13, 1e-16, 1e-17, 1e-18, 1e-19, 1e-20])
@pytest.mark.parametrize("eps", [1e-40, 1e-6])
def test_the_smallest_states(check, amp, eps):
    for _, fp64, ff, _, _ in check(2e-6, amp, eps):
        assert ff <= 1.03 * fp64


@pytest.mark.parametrize("amp", [1e-3, 1e-9, 1e-15, 1e-18, 1e-19, 1e-20, 1e-21])
def test_a_field_about_zero(check, amp):
    for _, _, _, _, worst in check(0.0, amp, 1e-40):
        assert worst <= 2.0 ** -40 * amp + 2.0 ** -94
