"""Factors of the integer A's epilogue outside the exponents it can form: the smoothed restriction
P^dagger (r - omega A r) with a damping of 1e-90 on fields down to the kernel's exponent range is
the restriction of the same field at order one, scaled (powers of two: exact up to the order of sums)."""
import numpy as np
import pytest

import workloads as W
from test_gpu_fixed_stencil import DEV, mg  # noqa: F401

torch = pytest.importorskip("torch")
pytestmark = pytest.mark.gpu


@pytest.mark.parametrize("omega", [1e-90, 1e-30, 0.02])
@pytest.mark.parametrize("power", [-800, -400, 700])
def test_scaled_fields(mg, omega, power):  # noqa: F811
    Lx, Lt, blocks, Nv = 16, 16, [(4, 4)], [4]
    U = torch.from_numpy(W.links_from_angles(W.quenched_u1_angles(Lx, Lt, 3.0, 2, 5))).to(DEV)
    noise = torch.from_numpy(W.setup_noise(Lx, Lt, blocks, Nv, 7)).to(DEV)
    r = torch.from_numpy(W.gaussian_field((1, Lt, Lx, 2), 3)).to(DEV)
    with mg.Multigrid(U, -0.5, blocks, Nv, noise, smooth_omega=omega) as s:
        out = []
        for scale in (1.0, 2.0 ** power):
            c = torch.empty((1, 4, 4, 8), dtype=torch.complex128, device=DEV)
            mg.mg_restrict(s.h, 1, r * scale, c, 1, mg.PREC_F64)
            out.append(c.cpu().numpy() / scale)
    assert np.all(np.abs(out[1] - out[0]) <= 1e-13 * np.abs(out[0]).max())
