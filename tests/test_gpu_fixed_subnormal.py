"""The integer FP64 A on fields of subnormal numbers alone, and of subnormal sites beside normal
ones: against extended precision.  A subnormal result carries the roundings of its FP64 sums, each
at most 2^-1075 and some 16 in a row sum, those of D psi multiplied by up to |4 + m| + 4 < 7 in the
second one: 200 units of 2^-1074."""
import numpy as np
import pytest

import workloads as W
from test_gpu_fixed_stencil import _apply, _wilson, mg  # noqa: F401

torch = pytest.importorskip("torch")
pytestmark = pytest.mark.gpu


@pytest.mark.parametrize("kind", ["all", "point", "beside"])
def test_subnormal_fields(mg, kind):  # noqa: F811
    Lx, Lt, mass = 44, 20, -2.0
    U = W.links_from_angles(W.quenched_u1_angles(Lx, Lt, 2.0, 2, 5))
    psi = W.gaussian_field((2, Lt, Lx, 2), 9) * 1e-309
    t, x = np.meshgrid(np.arange(Lt), np.arange(Lx), indexing="ij")
    if kind == "point":
        psi *= ((x == 3) & (t == 0))[None, :, :, None]
    elif kind == "beside":                               # half the lattice at order one
        psi[:, :, Lx // 2:] = W.gaussian_field((2, Lt, Lx // 2, 2), 10)
    y = _apply(mg, U, mass, psi, 2)
    diag = np.longdouble(4.0 + mass)
    ref = _wilson(U, diag, _wilson(U, diag, psi.astype(np.clongdouble), 1), -1)
    big = np.maximum(np.abs(psi.real), np.abs(psi.imag)).max(-1)
    loc = np.zeros_like(big)
    for dt in range(-2, 3):
        for dx in range(-2 + abs(dt), 3 - abs(dt)):
            loc = np.maximum(loc, np.roll(big, (dt, dx), (1, 2)))
    loc[loc < 1e-300] = 0.0                              # there the FP64 kernel's own roundings apply
    for part in (np.real, np.imag):
        err = np.abs(part(y).astype(np.longdouble) - part(ref))
        tol = diag ** 2 * 200 * 2.0 ** -58 * loc[..., None] + 2.0 ** -52 * np.abs(part(ref)) + 200 * np.longdouble(5e-324)
        assert np.all(err <= tol), float(np.max(err - tol))
    assert np.any(y[:, 2:18, 3:18] != 0) or kind == "point"
