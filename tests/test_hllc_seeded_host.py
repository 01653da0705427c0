"""CPU check of the FP64 HLLC flux with two-float seeds (hllc_seeded in face_ff.cuh), compiled for the host by
nvcc, against 80-bit arithmetic.  The flux is about 30 operations long, each with an error of 2^-53 of a
term of size (|u| + c) |U| (p for the pressure's), which the difference S - S* of size c magnifies by
at most (|u| + c) / c: every component stays within 32 of those units.  States outside the seeds' range
are refused."""
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
    exe = tmp_path_factory.mktemp("hllc") / "check_hllc_seeded"
    csrc = os.path.join(ROOT, "paper_2406_19494_gb300", "csrc")
    r = subprocess.run([nvcc, "-std=c++17", "-O2", "-Xcompiler", "-ffp-contract=off", "-diag-suppress", "177",
                        "-I" + csrc, "-I" + os.path.join(ROOT, "include"),
                        "-I" + os.path.join(ROOT, "paper_2406_19494_gb300", "include"),
                        os.path.join(ROOT, "tests", "native", "check_hllc_seeded.cu"), "-o", str(exe)],
                       capture_output=True, text=True)
    assert r.returncode == 0, r.stderr
    return lambda *a: subprocess.run([str(exe)] + [repr(float(x)) for x in a], capture_output=True, text=True).stdout.split()


@pytest.mark.parametrize("mach", [0.1, 1.0, 3.0, 20.0])
@pytest.mark.parametrize("jump", [0.02, 0.1, 0.6])
@pytest.mark.parametrize("scale", [1.0, 1e-8, 1e8])
def test_seeded_flux_is_exact_to_rounding(check, mach, jump, scale):
    taken, seeded, _ = check(mach, jump, scale)
    assert int(taken) == 100000 and float(seeded) <= 1.0


@pytest.mark.parametrize("scale", [1e-12, 1e12])
def test_states_outside_the_seeds_are_refused(check, scale):
    assert check(1.0, 0.1, scale)[0] == "0"
