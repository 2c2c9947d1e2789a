"""The integer FP64 coarse apply on vectors of subnormal numbers alone, and of such sites beside
normal ones, against the stored blocks in extended precision: 2^-49 of the sum of magnitudes as in
test_gpu_fixed_coarse, and 2^-1075 for each of the 4 FMAs of 9 n products and the 9 sums."""
import numpy as np
import pytest

import workloads as W
from test_gpu_fixed_coarse import _apply, _hierarchy, mg  # noqa: F401

torch = pytest.importorskip("torch")
pytestmark = pytest.mark.gpu


@pytest.mark.parametrize("kind", ["all", "point", "beside"])
@pytest.mark.parametrize("nrhs", [1, 6])
def test_subnormal_vectors(mg, nrhs, kind):  # noqa: F811
    n = 16
    s, A = _hierarchy(mg, 64, 32, n // 2)
    with s:
        x = W.gaussian_field((nrhs, 8, 8, n), 3) * 1e-310
        if kind == "point":
            keep = np.zeros((8, 8), bool)
            keep[3, 4] = True
            x[:, ~keep] = 0.0
        elif kind == "beside":
            x[:, :, 4:] = W.gaussian_field((nrhs, 8, 4, n), 4)
        y = _apply(mg, s, x)
    Al, xl = A.astype(np.clongdouble), x.astype(np.clongdouble)
    ref, mag, amp, row = np.zeros_like(xl), np.zeros(x.shape, np.longdouble), np.zeros(x.shape[:3]), 0.0
    for d in range(9):
        dx, dt = d % 3 - 1, d // 3 - 1
        xn = np.roll(xl, (-dt, -dx), (1, 2))
        ref += np.einsum("txab,rtxb->rtxa", Al[:, :, d], xn)
        mag += np.einsum("txab,rtxb->rtxa", np.abs(Al[:, :, d]), np.abs(xn))
        amp = np.maximum(amp, np.abs(xn).max(-1).astype(float))
        row = max(row, np.abs(A[:, :, d]).max())
    big = np.where(amp > 1e-300, amp, 0.0)[..., None]    # the integer sums' own tolerance, at normal sites
    tol = 2.0 ** -49 * mag + (36 * n + 9) * np.longdouble(5e-324) + 9 * 24 * n * 2.0 ** -56 * row * big
    assert np.all(np.abs(y - ref) <= tol), float(np.max(np.abs(y - ref) / tol))
    assert np.any(y[:, 2:5, 3:6] != 0)
