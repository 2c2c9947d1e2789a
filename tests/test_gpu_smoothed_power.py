"""The power iteration of a level below a smoothed coarsening: with a large damping and mass the
operator (1 - omega A) A (1 - omega A) there has norms of 10^10 and more, whose powers leave FP64
after 16 steps.  Its largest eigenvalue must come out, 0.9 of it at least after 30 steps; the norm is
at most (1 + omega a)^2 a with a = (|4 + m| + 4)^2."""
import pytest

import workloads as W

torch = pytest.importorskip("torch")
pytestmark = pytest.mark.gpu

DEV = "cuda:0"


@pytest.mark.parametrize("omega,mass", [(0.5, 60.0), (0.02, -0.5), (3.0, 20.0)])
def test_lambda_of_the_smoothed_level(omega, mass):
    if not torch.cuda.is_available():
        pytest.skip("no CUDA device")
    import __graft_entry__
    __graft_entry__.build()
    from paper_0710_3612_gb300 import mg
    L, blocks, Nv = 32, [(4, 4), (2, 2)], [4, 4]
    U = torch.from_numpy(W.links_from_angles(W.quenched_u1_angles(L, L, 6.0, 10, 1))).to(DEV)
    noise = torch.from_numpy(W.setup_noise(L, L, blocks, Nv, 7)).to(DEV)
    with mg.Multigrid(U, mass, blocks, Nv, noise, smooth_omega=omega) as s:
        lam = mg.mg_get_smoother(s.h, 2)[2]
        op = torch.empty((8, 8, 9, 8, 8), dtype=torch.complex128, device=DEV)
        mg.mg_get_coarse_op(s.h, 2, op)
    M = torch.zeros((64, 8, 64, 8), dtype=torch.complex128, device=DEV)
    j = torch.arange(64, device=DEV)
    for d in range(9):
        n = (j // 8 + d // 3 - 1) % 8 * 8 + (j % 8 + d % 3 - 1) % 8
        M[j, :, n, :] += op[:, :, d].reshape(64, 8, 8)
    top = torch.linalg.eigvalsh(M.reshape(512, 512))[-1].item()
    assert 0.9 * top <= lam <= top * (1 + 1e-10)
    a = (abs(4 + mass) + 4) ** 2
    assert top <= (1 + omega * a) ** 2 * a
