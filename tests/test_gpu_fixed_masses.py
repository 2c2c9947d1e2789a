"""The integer A at masses a rounding error away from a power of two of (4 + m)^2, as mass sweeps
reach them: plain, with the fused dot and inside the V-cycle's epilogues, then set-up, re-mass and
solve.  Plain results against extended precision (the tolerance of test_gpu_fixed_stencil); the
rest against the same calls at the round mass next to it, 1e-15 away: 1e-9 leaves a condition
number of 10^6 for it."""
import numpy as np
import pytest

import workloads as W
from test_gpu_fixed_stencil import DEV, _apply, _check, mg  # noqa: F401

torch = pytest.importorskip("torch")
pytestmark = pytest.mark.gpu

NEAR = [-2.0000000000000004, -2.0000000000000018, -2.0000000001, -4.5e-16]


@pytest.mark.parametrize("mass", NEAR)
def test_plain_and_dot(mg, mass):  # noqa: F811
    Lx, Lt = 40, 24
    U = W.links_from_angles(W.quenched_u1_angles(Lx, Lt, 2.0, 2, 5))
    psi = W.gaussian_field((3, Lt, Lx, 2), 8)
    y = _apply(mg, U, mass, psi, 3)
    _check(U, mass, psi, y)
    with mg.Multigrid(torch.from_numpy(U).to(DEV), mass, [], [], autotune=0) as s:
        x = torch.from_numpy(psi[0]).to(DEV)
        out, xAx = torch.empty_like(x), torch.zeros(2, dtype=torch.float64, device=DEV)
        mg.mg_apply_A_dot_noalloc(s.h, x, out, xAx)
        assert np.array_equal(out.cpu().numpy(), y[0])
        want = np.vdot(psi[0], y[0])
        assert want.real > 0 and abs(complex(*xAx.tolist()) - want) <= 1e-12 * abs(want)


def _close(a, b):
    return torch.linalg.vector_norm(a - b) <= 1e-9 * torch.linalg.vector_norm(b)


@pytest.mark.parametrize("mass,at", [(-2.0000000000000018, -2.0), (-4.5e-16, 0.0)])
def test_hierarchy(mg, mass, at):  # noqa: F811
    Lx, Lt, blocks, Nv = 32, 32, [(4, 4)], [4]
    U = torch.from_numpy(W.links_from_angles(W.quenched_u1_angles(Lx, Lt, 6.0, 10, 1))).to(DEV)
    noise = torch.from_numpy(W.setup_noise(Lx, Lt, blocks, Nv, 7)).to(DEV)
    b = torch.from_numpy(W.gaussian_field((Lt, Lx, 2), 3)).to(DEV)

    def results(s):
        z = torch.empty_like(b)
        mg.mg_vcycle(s.h, b, z, mg.PREC_F64)
        x, info = s.solve(b, tol=1e-12, solver=mg.SOLVER_MGCG_FP64)
        assert info[0].true_residual <= 1e-12
        return torch.tensor(list(mg.mg_get_smoother(s.h, 1)), dtype=torch.float64), z, x

    with mg.Multigrid(U, at, blocks, Nv, noise) as s:
        round_mass = results(s)
    with mg.Multigrid(U, mass, blocks, Nv, noise) as s:
        for got, want in zip(results(s), round_mass):
            assert _close(got, want)
    with mg.Multigrid(U, at, blocks, Nv, noise) as s:
        s.set_mass(mass)
        for got, want in zip(results(s)[1:], round_mass[1:]):
            assert _close(got, want)
