"""The integer FP64 A keeps the accuracy of small hop terms at every mass it takes: point sources and
fields that decay by 1 / (4 + m) per site, where the terms of a result are far smaller than the
largest component near it.  Tolerance per entry, of M = |D|^T |D| psi_max (psi_max the larger
component of a site, |D| the magnitudes of the stencil): a unit of a hop product is at most 12 of
2^-58 of its term; 18 units per D sum and 100 in the second one give 2^-47, and two FP64 roundings."""
import numpy as np
import pytest

import workloads as W
from test_gpu_fixed_stencil import _apply, _wilson, mg  # noqa: F401

torch = pytest.importorskip("torch")
pytestmark = pytest.mark.gpu


def _magnitudes(diag, big):
    """|D|^T |D| on site maxima: every hop adds both components over two."""
    for _ in range(2):
        big = diag * big + sum(np.roll(big, s, ax) for s in (-1, 1) for ax in (1, 2))
    return big


@pytest.mark.parametrize("mass", [-2.5, -2.0, -1.0, 0.0, 2.0, 7.9, 8.1, 28.0, 60.0, -5.5, -40.0])
@pytest.mark.parametrize("kind", ["point", "decay"])
def test_small_terms(mg, mass, kind):  # noqa: F811
    Lx, Lt = 44, 20
    U = W.links_from_angles(W.quenched_u1_angles(Lx, Lt, 2.0, 2, 5))
    psi = W.gaussian_field((2, Lt, Lx, 2), 9)
    t, x = np.meshgrid(np.arange(Lt), np.arange(Lx), indexing="ij")
    r = np.abs(x - 20) + np.abs(t - 10)
    psi *= (r == 0)[None, :, :, None] if kind == "point" else (abs(4 + mass) ** -r.astype(float))[None, :, :, None]
    y = _apply(mg, U, mass, psi, 2)
    diag = np.longdouble(4.0 + mass)
    ref = _wilson(U, diag, _wilson(U, diag, psi.astype(np.clongdouble), 1), -1)
    tol = 2.0 ** -47 * _magnitudes(abs(4 + mass), np.maximum(np.abs(psi.real), np.abs(psi.imag)).max(-1))[..., None]
    for part in (np.real, np.imag):
        err = np.abs(part(y).astype(np.longdouble) - part(ref))
        bound = tol + 2.0 ** -52 * np.abs(part(ref))
        assert np.all(err <= bound), float(np.max(err / np.maximum(bound, 1e-300)))
