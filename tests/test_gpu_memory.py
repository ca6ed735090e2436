"""Device memory of a handle: the digits of the sliced products fit in what a
handle of 14 (FP64) or 12 (split-BF16) tensors holds."""
import pytest

torch = pytest.importorskip("torch")
pytestmark = pytest.mark.gpu


@pytest.fixture(scope="module")
def fc():
    import __graft_entry__ as g
    g.build()
    from paper_2510_21394_gb300 import fcgle
    return fcgle


# tensors of 2 P reals per handle; both shapes run sliced products
@pytest.mark.parametrize("prec,ns,pad,real,tensors", [("fp64", [256, 240, 200], 4, 8, 14),
                                                      ("bf16x3", [264, 256, 300], 8, 4, 12)])
def test_handle_memory(fc, prec, ns, pad, real, tensors):
    def make(n):
        return fc.Solver(n, [(-4.0, 4.0)] * 3, [1.3, 1.7, 1.5], 1.0, 0.4, 0.5, 1.0, 0.2, precision=prec)

    def used():
        torch.cuda.synchronize()
        free, total = torch.cuda.mem_get_info()
        return total - free

    make([16, 264, 8]).close()   # the library's own one-time allocations
    p = [(n + pad - 1) // pad * pad for n in ns]
    P = p[0] * p[1] * p[2]
    before = used()
    s = make(ns)
    grew = used() - before
    s.close()
    # per direction, two matrices of at most 64 bytes an entry in all their forms (rows and
    # columns padded to 128), and 2 MB of rounding per allocation, at most 64 of them
    matrices = sum(2 * 64 * ((q + 127) // 128 * 128) ** 2 for q in p)
    assert grew <= tensors * 2 * P * real + matrices + 64 * (2 << 20)
