"""What the kernel sources may not contain."""
import glob
import os

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
