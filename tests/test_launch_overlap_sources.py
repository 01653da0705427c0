"""Kernels that begin before the kernel that writes their input has ended (launch_step in fluid_internal.cuh)
keep three rules, read from the sources: their first statement is the wait, none of their pointer parameters
is __restrict__ (the compiler may move such loads ahead of the wait, or take the read-only load path, which
is not defined for data written during the kernel's lifetime), and no function they can reach reads another
kernel's output by __ldg."""
import os
import re

from conftest import ROOT

CSRC = os.path.join(ROOT, "paper_2406_19494_gb300", "csrc")


def _sources():
    for f in sorted(os.listdir(CSRC)):
        if f.endswith((".cu", ".cuh")):
            s = open(os.path.join(CSRC, f)).read()
            yield f, re.sub(r"//[^\n]*", "", s)


def test_overlapped_kernels_wait_first_and_load_plainly():
    launched, kernels = set(), {}
    for f, s in _sources():
        launched |= set(re.findall(r"launch_step\((k_\w+)", s))
        for m in re.finditer(r"__global__", s):
            head, body = s[m.start():].split("{", 1)
            kernels[re.findall(r"(k[bm]*_\w+|kbm_\w+)\(", head)[-1]] = (f, head, body.lstrip())
    launched.discard("kernel")
    launched |= {"k_face_mixed_x", "k_face_mixed_t"}       # launch_t picks one of the two by axis
    assert len(launched) >= 20 and launched <= set(kernels)
    for k in launched:
        f, head, body = kernels[k]
        assert body.startswith("step_wait();"), (f, k)
        assert "__restrict__" not in head, (f, k)


def test_the_read_only_load_stays_with_plain_launches():
    for f, s in _sources():
        if f == "kernels_adjoint.cu":
            # k_adj_face and what only it calls come before the overlapped kernels of the file
            s = s[s.index("k_adj_gather("):]
        assert not re.findall(r"__ldg\((?!g\.mf32)[^\n]*", s), f
