"""The tcgen05 coarsest product itself against the product in 64 bits (the solves refine its errors
away): tile rows that do not fill a CTA, padded rows, right-hand-side remainders, accumulation and
the FP32 copy.

Tolerance, of the sum of magnitudes S = |B| |x|: a product of split operands is exact to 3 units of
2^-22 (each low word to 2^-23, low times low left out); a column block adds 3 x 128 products and
up to 64 blocks are added in FP32: (384 + 64) / 2^24 at most.  Below 2^-15 in all.  The second
test's operands differ from TF32 numbers by 2^-12 of themselves, all the same way: without their
low words it misses by 2^-12, twice."""
import ctypes

import pytest

torch = pytest.importorskip("torch")
pytestmark = pytest.mark.gpu

DEV = "cuda:0"
P, I = ctypes.c_void_p, ctypes.c_int


@pytest.fixture(scope="module")
def lib():
    if not torch.cuda.is_available():
        pytest.skip("no CUDA device")
    import __graft_entry__
    __graft_entry__.build()
    return ctypes.CDLL(__graft_entry__.LIB)


def _product(lib, B, x, y=None):
    """(y +) B x by the kernel, in FP64 and as its FP32 copy; B [N][N] complex64, x [nrhs][N]."""
    N, nrhs = B.shape[0], x.shape[0]
    ld = (N + 63) // 64 * 64
    M = torch.zeros((ld, ld), dtype=torch.complex64, device=DEV)
    M[:N, :N] = B
    nt = ld // 64
    packed = torch.zeros(nt * (nt + 1) // 2 * 4096, dtype=torch.complex64, device=DEV)
    scratch = torch.zeros((nrhs, ld), dtype=torch.complex64, device=DEV)
    part = torch.zeros(nt * 2 * nrhs * ld, dtype=torch.float32, device=DEV)
    out = torch.zeros_like(x) if y is None else y.clone()
    out32 = torch.zeros(x.shape, dtype=torch.complex64, device=DEV)
    s = P(torch.cuda.current_stream().cuda_stream)
    assert lib._ZN3mgk14pack_hermitianEPKvPviP11CUstream_st(P(M.data_ptr()), P(packed.data_ptr()), I(ld), s) == 0
    assert lib._ZN3mgk17hermitian_gemv_tcEPKvS1_PviiiS2_S2_bS2_P11CUstream_st(
        P(packed.data_ptr()), P(x.data_ptr()), P(out.data_ptr()), I(N), I(ld), I(nrhs), P(scratch.data_ptr()),
        P(part.data_ptr()), ctypes.c_bool(y is not None), P(out32.data_ptr()), s) == 0
    flag = I(0)
    assert lib._ZN3mgk18gemv_tc_take_errorEPi(ctypes.byref(flag)) == 0 and flag.value == 0
    return out, out32


def _check(lib, B, x, y=None):
    out, out32 = _product(lib, B, x, y)
    xs = x.to(torch.complex64).to(torch.complex128)
    ref = xs @ B.to(torch.complex128).T + (0 if y is None else y)
    S = xs.abs() @ B.to(torch.complex128).abs().T
    assert torch.all((out - ref).abs() <= 2.0 ** -15 * S)
    assert torch.equal(out32, out.to(torch.complex64))


@pytest.mark.parametrize("N,nrhs", [(64, 16), (100, 17), (192, 33), (1000, 64), (1024, 40), (4096, 16), (2000, 64)])
def test_random_hermitian(lib, N, nrhs):
    g = torch.Generator(device=DEV)
    g.manual_seed(N + nrhs)
    B = torch.view_as_complex(torch.randn((N, N, 2), generator=g, device=DEV))
    B = torch.tril(B, -1)
    B = B + B.conj().T + torch.diag(torch.randn(N, generator=g, device=DEV)).to(torch.complex64)
    x = torch.view_as_complex(torch.randn((nrhs, N, 2), generator=g, device=DEV, dtype=torch.float64))
    _check(lib, B, x)
    _check(lib, B, x, x.flip(0).contiguous())


@pytest.mark.parametrize("N,nrhs", [(200, 16), (1024, 64)])
def test_low_words_count(lib, N, nrhs):
    B = torch.full((N, N), 1 + 2.0 ** -12, dtype=torch.complex64, device=DEV)
    x = torch.full((nrhs, N), 1 + 2.0 ** -12, dtype=torch.complex128, device=DEV)
    _check(lib, B, x)
