"""The FP32 reductions of the reliable solver keep single precision per entry and double beyond, in
batches as with one right-hand side: sums in which small entries follow a large one in the same
thread.  An entry's two products round twice (2 units of 2^-24 of their magnitudes; the sums here
are built of exact products, so 2^-40 covers the FP64 additions); chains in FP32 would lose the
small entries, 1.7e-8 each of the large one."""
import ctypes

import pytest

torch = pytest.importorskip("torch")
pytestmark = pytest.mark.gpu

DEV = "cuda:0"
P, LL, I, D = ctypes.c_void_p, ctypes.c_longlong, ctypes.c_int, ctypes.c_double


@pytest.fixture(scope="module")
def lib():
    if not torch.cuda.is_available():
        pytest.skip("no CUDA device")
    import __graft_entry__
    __graft_entry__.build()
    return ctypes.CDLL(__graft_entry__.LIB)


def _ptr(t):
    return P(t.data_ptr())


def _ws(nrhs):
    return torch.zeros(64 + 2 * 608 * nrhs, dtype=torch.float64, device=DEV)


def _stream():
    return P(torch.cuda.current_stream().cuda_stream)


@pytest.mark.parametrize("count,nrhs", [(16384, 64), (131072, 64), (131072, 8), (1 << 20, 1), (777, 3)])
def test_reductions(lib, count, nrhs):
    v = torch.full((nrhs, count), 2.0 ** -13, dtype=torch.complex64, device=DEV)
    v[:, :256] = 1.0                                     # the first entry of some threads
    want = torch.sum(torch.abs(v.to(torch.complex128)) ** 2, -1)
    out = torch.zeros((nrhs, 2), dtype=torch.float64, device=DEV)
    lib._ZN3mgk4rdotEPKvS1_xiPdS2_P11CUstream_st(_ptr(v), _ptr(v), LL(count), I(nrhs), _ptr(_ws(nrhs)), _ptr(out),
                                                 _stream())
    assert torch.all(torch.abs(out[:, 0] - want) <= 2.0 ** -40 * want) and torch.all(out[:, 1] == 0)
    lib._ZN3mgk11rdot2_zq_rzEPKvS1_S1_xiPdS2_P11CUstream_st(_ptr(v), _ptr(v), _ptr(v), LL(count), I(nrhs),
                                                            _ptr(_ws(nrhs)), _ptr(out), _stream())
    assert torch.all(torch.abs(out - want[:, None]) <= 2.0 ** -40 * want[:, None])
    x, r = torch.zeros_like(v), v.clone()
    one, zero = torch.ones((nrhs, 2), dtype=torch.float64, device=DEV), torch.zeros((nrhs, 2), dtype=torch.float64, device=DEV)
    lib._ZN3mgk6rcg_xrEPvS0_PKvS2_PKdS4_PKixiPdS7_P11CUstream_st(
        _ptr(x), _ptr(r), _ptr(v), _ptr(v), _ptr(zero), _ptr(one), P(None), LL(count), I(nrhs), _ptr(_ws(nrhs)),
        _ptr(out), _stream())                            # alpha = 0: |r|^2 alone
    assert torch.all(torch.abs(out[:, 0] - want) <= 2.0 ** -40 * want)


def test_fused_dot_over_two_rows(lib):
    """Tiles of 32 x 16 give a thread the rows t and t + 8; the two point sources do not touch."""

    class Epilogue(ctypes.Structure):
        _fields_ = [("ca", D), ("cu", D), ("cw", D), ("U", P), ("W", P), ("ws", P), ("out", P), ("real", ctypes.c_bool),
                    ("q", P), ("r", P)]

    L, nrhs = 64, 64
    U = torch.ones((2, L, L), dtype=torch.complex64, device=DEV)
    x = torch.zeros((nrhs, L, L, 2), dtype=torch.complex64, device=DEV)
    x[:, 17, 37, 0], x[:, 25, 37, 0] = 1.0, 2.0 ** -13
    y, out = torch.empty_like(x), torch.zeros((nrhs, 2), dtype=torch.float64, device=DEV)
    ws = _ws(nrhs)
    ep = Epilogue(1.0, 0.0, 0.0, None, None, ws.data_ptr(), out.data_ptr(), False, None, None)
    e = lib._ZN3mgk8wilson_AIfEE9cudaErrorPKvPvS3_S3_diiiRKNS_8EpilogueEP11CUstream_st(
        _ptr(x), _ptr(y), _ptr(U), P(None), D(2.0), I(L), I(L), I(nrhs), ctypes.byref(ep), _stream())
    assert e == 0
    want = torch.sum((x.to(torch.complex128).conj() * y.to(torch.complex128)).real, (1, 2, 3))
    assert want[0].item() > 1 and torch.equal(out[:, 0], want)   # two exact products, added in FP64
