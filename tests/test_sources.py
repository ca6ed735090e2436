"""What the kernel sources may not contain."""
import glob
import os
import re

CSRC = os.path.join(os.path.dirname(os.path.dirname(os.path.abspath(__file__))), "paper_2510_21394_gb300", "csrc")


def test_no_multicast_loads():
    # the same kernels run in the multi-process paths (one process per GPU), which
    # use no TMA multicast: no load or commit names a multicast form
    files = glob.glob(os.path.join(CSRC, "*.cu*")) + glob.glob(os.path.join(CSRC, "*.h"))
    assert files
    for f in files:
        with open(f) as fh:
            assert "multicast::cluster" not in fh.read(), os.path.basename(f)


def test_setup_uploads_follow_the_stream():
    # a plain cudaMemcpy runs on the legacy default stream, which non-blocking
    # streams (a batch's) do not wait for: host data reaches a handle by upload()
    files = glob.glob(os.path.join(CSRC, "*.cu*")) + glob.glob(os.path.join(CSRC, "*.cpp"))
    for f in files:
        with open(f) as fh:
            for line in fh:
                assert not ("cudaMemcpy(" in line and "cudaMemcpyHostToDevice" in line), (os.path.basename(f), line)


def _parameters(src, start):
    """The parameter list of a __global__ function that begins at `start`, and its body."""
    def closing(i, a, b):
        depth = 0
        for j in range(i, len(src)):
            depth += (src[j] == a) - (src[j] == b)
            if depth == 0:
                return j
        raise ValueError("unbalanced")
    i = src.index("(", start)
    if "__launch_bounds__" in src[start:i]:
        i = src.index("(", closing(i, "(", ")"))
    j = closing(i, "(", ")")
    b = src.index("{", j)
    return src[i:j], src[b:closing(b, "{", "}")]


def test_dependent_kernels_read_no_results_through_the_read_only_path():
    # a dependent kernel lives while its predecessors still write: its inputs are no
    # const __restrict__ parameters; exponents of the handle's matrices and the
    # descriptors of a batch are constants
    constants = {"em", "gd"}
    found = 0
    for f in glob.glob(os.path.join(CSRC, "*.cu*")):
        with open(f) as fh:
            src = re.sub(r"//.*", "", fh.read())
        for m in re.finditer(r"__global__ void", src):
            params, body = _parameters(src, m.end())
            if "pdl_wait()" not in body and "pdl_enter()" not in body:
                continue
            found += 1
            bad = [n for n in re.findall(r"const [\w:<>]+\s*\* __restrict__ (\w+)", params) if n not in constants]
            assert not bad, (os.path.basename(f), params, bad)
    assert found >= 20
