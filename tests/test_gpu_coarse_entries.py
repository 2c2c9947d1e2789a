"""The integer FP64 coarse apply where a vector's largest component meets none but small entries:
one component per right-hand side on every third site, against a hierarchy of mass 60, whose
blocks hold off-diagonal entries 2^-10 of the diagonal and smaller.  A row is one product here.  In
integers it is exact to 24 units of 2^-56 of largest times largest, which is at most 2^8 of the
product's magnitude (smaller rows take the FP64 path): 24 units of 2^-48."""
import numpy as np
import pytest

import workloads as W
from test_gpu_fixed_coarse import DEV, _apply, mg  # noqa: F401

torch = pytest.importorskip("torch")
pytestmark = pytest.mark.gpu


def test_unit_vectors(mg):  # noqa: F811
    Lx, Lt, n = 96, 48, 16
    U = W.links_from_angles(W.quenched_u1_angles(Lx, Lt, 3.0, 2, 5))
    noise = torch.from_numpy(W.setup_noise(Lx, Lt, [(8, 4)], [n // 2], 7)).to(DEV)
    with mg.Multigrid(torch.from_numpy(U).to(DEV), 60.0, [(8, 4)], [n // 2], noise, autotune=0) as s:
        At = torch.empty((Lt // 4, Lx // 8, 9, n, n), dtype=torch.complex128, device=DEV)
        mg.mg_get_coarse_op(s.h, 2, At)
        A = At.cpu().numpy()
        x = np.zeros((n, Lt // 4, Lx // 8, n), dtype=np.complex128)
        for c in range(n):
            x[c, ::3, ::3, c] = 1.0 / 3.0 - 2.0j / 7.0
        y = _apply(mg, s, x)
        one = _apply(mg, s, x[3:4].copy())
    assert np.array_equal(one[0], y[3])
    ref, mag = np.zeros_like(x), np.zeros(x.shape)
    for d in range(9):
        xn = np.roll(x, (1 - d // 3, 1 - d % 3), (1, 2))
        ref += np.einsum("txab,rtxb->rtxa", A[:, :, d], xn)
        mag += np.einsum("txab,rtxb->rtxa", np.abs(A[:, :, d]), np.abs(xn))
    assert np.all(np.abs(y - ref) <= 24 * 2.0 ** -48 * mag), float(np.max(np.abs(y - ref) / mag))
