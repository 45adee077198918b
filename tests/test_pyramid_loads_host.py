"""The pyramid kernels start while the launch before them still writes the
level they read (programmatic dependent launch): they read pixels by ordinary
loads, never through the read-only path, and a kernel launched that way waits
before its first one."""

import os
import re

CSRC = os.path.join(os.path.dirname(os.path.dirname(os.path.abspath(__file__))), "paper_2607_01757_gb300", "csrc")


def _code(name):
    with open(os.path.join(CSRC, name)) as f:
        return re.sub(r"//[^\n]*", "", f.read())


def test_no_read_only_loads_of_pixels():
    src = _code("vt_pyramid.cu")
    assert not re.search(r"__ldg|ld\.global\.nc|ld\.global\.[\w.]*\bnc\b|__restrict__", src)


def test_dependent_kernels_wait():
    for name in sorted(os.listdir(CSRC)):
        if not name.endswith(".cu"):
            continue
        src = _code(name)
        for k in set(re.findall(r"launch_pdl\(\s*(k_\w+)", src)) | {m for m in re.findall(r"\bk_pyr\w*", src)}:
            bodies = [b for b in re.findall(r"__global__[^;{]*\b" + k + r"\([^{]*\{(.*?)\n\}", src, re.S)]
            assert all("pdl_wait()" in b for b in bodies), (name, k)
