"""Rules of the kernels that are set up while their predecessor still writes their inputs (launch_dep,
csrc/common.cuh), read from the sources: every such kernel waits for the predecessor (grid_dep), and
none reads global memory as read-only data (__ldg, or a const __restrict__ pointer, whose loads the
compiler may make non-coherent and move past the wait)."""
import glob
import os
import re

ROOT = os.path.dirname(os.path.dirname(os.path.abspath(__file__)))
CSRC = os.path.join(ROOT, "paper_2411_09287_gb300", "csrc")


def _sources():
    out = {}
    for path in sorted(glob.glob(os.path.join(CSRC, "*.cu")) + glob.glob(os.path.join(CSRC, "*.cuh"))):
        src = re.sub(r"/\*.*?\*/", "", open(path).read(), flags=re.S)
        out[os.path.basename(path)] = re.sub(r"//[^\n]*", "", src)
    return out


def _kernels(src):
    """(name, body) of every __global__ function."""
    for m in re.finditer(r"__global__\s", src):
        i = src.index("{", m.end())
        head = re.sub(r"__launch_bounds__\((?:[^()]|\([^()]*\))*\)", "", src[m.end():i])
        name = re.search(r"(\w+)\s*\(", head).group(1)
        depth, j = 1, i + 1
        while depth:
            depth += {"{": 1, "}": -1}.get(src[j], 0)
            j += 1
        yield name, src[i:j]


def test_no_read_only_loads():
    for name, src in _sources().items():
        for bad in (r"__ldg\s*\(", r"ld\.global\.nc", r"const\s+[\w ]+\*\s*__restrict__"):
            assert not re.search(bad, src), (name, bad, re.search(bad, src).group(0))


def test_dependent_kernels_wait():
    seen = 0
    for name, src in _sources().items():
        assert "<<<" not in src, name   # launch_dep sets the launch up, and counts it
        for kernel, body in _kernels(src):
            seen += 1
            assert "grid_dep();" in body, kernel
    assert seen > 50
