"""Coarsest-level product for 16 to 64 right-hand sides on tcgen05 (3 x TF32), at the
edges of its range and tiles: the smallest levels that take it, an odd number of tile rows
(the last block of 128 rows half empty), a ragged last tile, right-hand sides that do not
fill a group of 8.

One iteration of the FP64 multigrid CG on each right-hand side of a batch against the
same iteration alone (whose product runs in FP32 FMAs).  Both refine the coarsest solve in
FP64 to a relative residual of coarsest_tol = 1e-12, so they may differ by twice the
condition number times that; at m = 0.1, A's spectrum lies in [0.1^2, 8.1^2] and Galerkin
projection keeps it there: 2 * 6.6e3 * 1e-12."""
import numpy as np
import pytest

import workloads as W

torch = pytest.importorskip("torch")
pytestmark = pytest.mark.gpu

DEV = "cuda:0"
TOL = 2 * 6.6e3 * 1e-12


@pytest.fixture(scope="module")
def mg():
    if not torch.cuda.is_available():
        pytest.skip("no CUDA device")
    import __graft_entry__
    __graft_entry__.build()
    from paper_0710_3612_gb300 import mg as m
    return m


@pytest.mark.parametrize("Lx,Lt,nrhs", [(64, 16, 64), (68, 16, 64), (52, 20, 64), (48, 44, 33), (64, 64, 16),
                                        (64, 64, 23)])
def test_batch_equals_single(mg, Lx, Lt, nrhs):
    blocks, Nv = [(4, 4)], [8]                       # Lx Lt unknowns in tiles of 64
    U = torch.from_numpy(W.quenched_u1(Lx, Lt, 6.0, 20, 3)).to(DEV)
    noise = torch.from_numpy(W.setup_noise(Lx, Lt, blocks, Nv, 5)).to(DEV)
    b = torch.from_numpy(np.stack([W.gaussian_field((Lt, Lx, 2), 300 + k) for k in range(nrhs)])).to(DEV)
    with mg.Multigrid(U, 0.1, blocks, Nv, noise, max_rhs=nrhs, coarsest_tol=1e-12) as s:
        x, _ = s.solve(b, tol=1e-30, maxiter=1, solver=mg.SOLVER_MGCG_FP64)
    with mg.Multigrid(U, 0.1, blocks, Nv, noise, coarsest_tol=1e-12) as s:
        for k in range(nrhs):
            y, _ = s.solve(b[k].contiguous(), tol=1e-30, maxiter=1, solver=mg.SOLVER_MGCG_FP64)
            assert (torch.linalg.vector_norm(x[k] - y) <= TOL * torch.linalg.vector_norm(y)).item(), k
