"""The sparsity-ordered dense inverse of the coarsest level: one block, padded sizes, sites that
straddle 64-row blocks, coarse extents of 2 (couplings that alias), thin lattices with many
independent pivots.  The refined solve must reach its residual (coarsest_tol = 1e-13; 1e-12 leaves
room for the FP64 rounding of the residual at condition numbers near 10) on the stored operator,
with at most one refinement step more than the inversion that sweeps every block in order."""
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


@pytest.mark.parametrize("Lx,Lt,Nv", [(8, 8, 2), (8, 8, 8), (16, 32, 5), (64, 8, 4), (8, 128, 8), (40, 24, 12), (64, 64, 8)])
def test_inverse_against_the_operator(mg, Lx, Lt, Nv):
    U = torch.from_numpy(W.links_from_angles(W.quenched_u1_angles(Lx, Lt, 3.0, 2, 5))).to(DEV)
    noise = torch.from_numpy(W.setup_noise(Lx, Lt, [(4, 4)], [Nv], 7)).to(DEV)
    lx, lt, n = Lx // 4, Lt // 4, 2 * Nv
    steps = {}
    for tc in (0, 1):
        with mg.Multigrid(U, 0.0, [(4, 4)], [Nv], noise, autotune=0, coarsest_gj_tcgen05=tc) as s:
            dense, steps[tc], res = mg.mg_get_coarsest_info(s.h)
            assert dense and res <= 1e-13
            b = W.gaussian_field((lt, lx, n), 3)
            x = torch.empty((lt, lx, n), dtype=torch.complex128, device=DEV)
            mg.mg_coarsest_solve(s.h, torch.from_numpy(b).to(DEV), x)
            A = torch.empty((lt, lx, 9, n, n), dtype=torch.complex128, device=DEV)
            mg.mg_get_coarse_op(s.h, 2, A)
            A, x = A.cpu().numpy(), x.cpu().numpy()
            r = b.copy()
            for d in range(9):
                r -= np.einsum("txab,txb->txa", A[:, :, d], np.roll(x, (1 - d // 3, 1 - d % 3), (0, 1)))
            assert np.linalg.norm(r) <= 1e-12 * np.linalg.norm(b)
    assert steps[0] <= steps[1] + 1
