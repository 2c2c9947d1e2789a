"""The integer-arithmetic A = D^dagger D on FP64 vectors: every tile edge, right-hand-side
count and mass at the limits of its range against extended precision, with fields of huge
dynamic range, point sources, denormals, infinities and NaN.

Tolerance per entry: 100 units of 2^-58 of the largest component within two hops (each unit at
most twice that component), from one unit per truncation: 1 for a converted component, 4 per hop
product (|w| <= 1/3), 18 per D sum, 20 per product and 99 per sum of the second application; and
two FP64 roundings of the result."""
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


def _wilson(U, diag, psi, s):
    """D (s = 1) or D^dagger (s = -1) in extended precision; psi[rhs][t][x][2]."""
    u = U.astype(np.clongdouble)
    u[1, -1] *= -1
    out = diag * psi
    for mu, ax in ((0, 2), (1, 1)):
        up = u[mu][None] * np.roll(psi, -1, axis=ax).transpose(3, 0, 1, 2)
        dn = np.roll(np.conj(u[mu])[None, :, :, None] * psi, 1, axis=ax).transpose(3, 0, 1, 2)
        one = 1 if mu == 0 else -1j
        for (f0, f1), sg in ((up, s), (dn, -s)):
            h = f0 - sg * f1 if mu == 0 else f0 + 1j * sg * f1
            out[..., 0] -= h / 2
            out[..., 1] -= h / 2 * (-sg * one if mu == 0 else sg * one)
    return out


def _check(U, mass, psi, y):
    diag = np.longdouble(4.0 + mass)
    p = psi.astype(np.clongdouble)
    ref = _wilson(U, diag, _wilson(U, diag, p, 1), -1)
    big = np.maximum(np.abs(psi.real), np.abs(psi.imag)).max(-1)
    loc = np.zeros_like(big)
    for dt in range(-2, 3):
        for dx in range(-2 + abs(dt), 3 - abs(dt)):
            loc = np.maximum(loc, np.roll(big, (dt, dx), (1, 2)))
    for part in (np.real, np.imag):
        err = np.abs(part(y).astype(np.longdouble) - part(ref))
        tol = diag ** 2 * 200 * 2.0 ** -58 * loc[..., None] + 2.0 ** -52 * np.abs(part(ref))
        assert np.all(err <= tol), float(np.max(err - tol))


def _apply(mg, U, mass, psi, nrhs):
    Lt, Lx = U.shape[1:]
    with mg.Multigrid(torch.from_numpy(U).to(DEV), mass, [], [], autotune=0) as s:
        x = torch.from_numpy(psi).to(DEV)
        y = torch.empty_like(x)
        mg.mg_apply_A(s.h, x, y, nrhs, mg.PREC_F64)
        return y.cpu().numpy()


@pytest.mark.parametrize("Lx,Lt,nrhs,mass", [
    (4, 4, 1, -2.0), (16, 8, 3, -2.5), (18, 10, 64, -2.07), (34, 18, 5, 0.1), (96, 130, 6, -2.0), (256, 258, 4, -1.9),
    (32, 16, 1, 60.0), (32, 16, 2, -6.0), (32, 16, 2, -2.51), (32, 16, 2, 60.5)])
def test_tiles_and_masses(mg, Lx, Lt, nrhs, mass):
    U = W.links_from_angles(W.quenched_u1_angles(Lx, Lt, 2.0, 2, 5))
    psi = W.gaussian_field((nrhs, Lt, Lx, 2), 8)
    _check(U, mass, psi, _apply(mg, U, mass, psi, nrhs))


@pytest.mark.parametrize("kind", ["range", "decay", "point", "tiny", "huge", "free"])
def test_fields(mg, kind):
    Lx, Lt = 44, 20
    U = W.links_from_angles(W.quenched_u1_angles(Lx, Lt, 2.0, 2, 5))
    psi = W.gaussian_field((1, Lt, Lx, 2), 9)
    rng = np.random.default_rng(1)
    t, x = np.meshgrid(np.arange(Lt), np.arange(Lx), indexing="ij")
    if kind == "range":                                  # site magnitudes over 2^+-300
        psi *= 2.0 ** rng.integers(-300, 300, (1, Lt, Lx, 1))
    elif kind == "decay":
        psi *= np.exp(-2.0 * np.hypot(x - 20, t - 10))[None, :, :, None]
    elif kind == "point":
        psi *= ((x == 3) & (t == 0))[None, :, :, None]
    elif kind == "tiny":                                 # below the kernel's exponent range
        psi *= 1e-290
    elif kind == "huge":
        psi *= 1e290
    else:                                                # unit links: the words of 1 / (2 diag)
        U = np.ones_like(U)
        psi = np.round(psi * 4)
    _check(U, -2.0, psi, _apply(mg, U, -2.0, psi, 1))


@pytest.mark.parametrize("bad", [np.inf, -np.inf, np.nan])
def test_non_finite(mg, bad):
    Lx, Lt = 40, 24
    U = W.links_from_angles(W.quenched_u1_angles(Lx, Lt, 2.0, 2, 5))
    psi = W.gaussian_field((1, Lt, Lx, 2), 9)
    clean = _apply(mg, U, -2.0, psi, 1)
    psi[0, 0, 39, 1] = bad
    y = _apply(mg, U, -2.0, psi, 1)
    t, x = np.meshgrid(np.arange(Lt), np.arange(Lx), indexing="ij")
    near = np.minimum(t, Lt - t) + np.minimum(np.abs(x - 39), Lx - np.abs(x - 39)) <= 2
    # two hops along one axis cancel exactly, but inf - inf does not: as in floating point
    assert not np.any(np.isfinite(y[0][near]).all(-1))
    assert np.array_equal(y[0][~near], clean[0][~near])
