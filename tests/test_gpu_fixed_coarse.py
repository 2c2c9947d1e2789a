"""The integer-arithmetic FP64 coarse apply: dof counts up to and above its limit (32), one and
several right-hand sides with every remainder of its groups of four, coarse extents of 2, vectors
of huge dynamic range, zeros, infinities and NaN, against the stored blocks applied in numpy.

Tolerance per entry: a row of n entries is exact to 24 units of 2^-56 per entry (two truncated
operands in three real products) of its largest entry times the largest component of its x(j + d);
nine rows, and 2^-49 of the sum of magnitudes for both sides' FP64 roundings."""
import numpy as np
import pytest

import workloads as W

torch = pytest.importorskip("torch")
pytestmark = pytest.mark.gpu

DEV = "cuda:0"


@pytest.fixture(scope="module")
def mg():
    if not torch.cuda.is_available():
        pytest.skip("no CUDA device")
    import __graft_entry__
    __graft_entry__.build()
    from paper_0710_3612_gb300 import mg as m
    return m


def _hierarchy(mg, Lx, Lt, Nv):
    U = W.links_from_angles(W.quenched_u1_angles(Lx, Lt, 3.0, 2, 5))
    noise = torch.from_numpy(W.setup_noise(Lx, Lt, [(8, 4)], [Nv], 7)).to(DEV)
    s = mg.Multigrid(torch.from_numpy(U).to(DEV), -1.9, [(8, 4)], [Nv], noise, autotune=0)
    A = torch.empty((Lt // 4, Lx // 8, 9, 2 * Nv, 2 * Nv), dtype=torch.complex128, device=DEV)
    mg.mg_get_coarse_op(s.h, 2, A)
    return s, A.cpu().numpy()


def _apply(mg, s, x):
    xt = torch.from_numpy(x).to(DEV)
    y = torch.empty_like(xt)
    mg.mg_apply_coarse(s.h, 2, xt, y, x.shape[0], mg.PREC_F64)
    return y.cpu().numpy()


def _check(A, x, y):
    ref, tol = np.zeros_like(x), np.zeros(x.shape)
    amp = np.maximum(np.abs(x.real), np.abs(x.imag)).max(-1)
    row = np.maximum(np.abs(A.real), np.abs(A.imag)).max(-1)
    for d in range(9):
        dx, dt = d % 3 - 1, d // 3 - 1
        xn = np.roll(x, (-dt, -dx), (1, 2))
        ref += np.einsum("txab,rtxb->rtxa", A[:, :, d], xn)
        tol += 24 * x.shape[-1] * 2.0 ** -56 * row[None, :, :, d] * np.roll(amp, (-dt, -dx), (1, 2))[..., None]
        tol += 2.0 ** -49 * np.einsum("txab,rtxb->rtxa", np.abs(A[:, :, d]), np.abs(xn))
    err = np.abs(y - ref)
    assert np.all(err <= tol), float(np.max(err / np.maximum(tol, 1e-300)))


@pytest.mark.parametrize("Lx,Lt,Nv,nrhs", [
    (16, 8, 1, 1), (16, 8, 4, 3), (32, 16, 8, 1), (32, 16, 8, 2), (48, 24, 8, 64), (40, 12, 12, 5), (32, 16, 12, 1),
    (32, 16, 16, 7), (32, 16, 16, 1), (32, 16, 20, 2)])
def test_against_blocks(mg, Lx, Lt, Nv, nrhs):
    s, A = _hierarchy(mg, Lx, Lt, Nv)
    with s:
        x = W.gaussian_field((nrhs, Lt // 4, Lx // 8, 2 * Nv), 3)
        _check(A, x, _apply(mg, s, x))


@pytest.mark.parametrize("nrhs", [1, 6])
def test_ranges(mg, nrhs):
    s, A = _hierarchy(mg, 64, 32, 8)
    rng = np.random.default_rng(2)
    with s:
        x = W.gaussian_field((nrhs, 8, 8, 16), 3)
        wide = x * 2.0 ** rng.integers(-60, 60, (nrhs, 8, 8, 1))
        _check(A, wide, _apply(mg, s, wide))
        point = np.zeros_like(x)
        point[:, 3, 4, 5] = 1.0 - 2.0j
        y = _apply(mg, s, point)
        _check(A, point, y)
        assert np.count_nonzero(np.abs(y).max(-1)) == 9 * nrhs
        for scale in (1e-250, 1e250):                    # outside the exponent range: the FP64 path
            _check(A, x * scale, _apply(mg, s, x * scale))
        clean = _apply(mg, s, x)
        for bad in (np.inf, np.nan):
            z = x.copy()
            z[0, 2, 2, 7] = bad
            y = _apply(mg, s, z)
            assert not np.any(np.isfinite(y[0, 1:4, 1:4]))
            far = np.ones((8, 8), bool)
            far[1:4, 1:4] = False
            assert np.array_equal(y[0][far], clean[0][far]) and np.array_equal(y[1:], clean[1:])
