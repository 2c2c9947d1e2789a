"""The FP32 streaming stencil (two sites per lane): lattices whose last strip of 60 sites is full,
one pair wide or partial, row blocks with remainders, batches, and the smoother's epilogue with
the output aliasing its operand, against the FP64 stencil.

Tolerance: A is 45 FP32 roundings deep at most (two hops of a product, sums of five terms and a
scaling each, operands rounded once), each 2^-24 of at most (|4 + m| + 4)^2 times the largest
component within two hops."""
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


@pytest.mark.parametrize("Lx,Lt,nrhs", [(120, 32, 64), (122, 24, 64), (178, 18, 64), (64, 1024, 30), (1024, 256, 4), (256, 250, 33)])
def test_streaming_stencil(mg, Lx, Lt, nrhs):
    U = torch.from_numpy(W.links_from_angles(W.quenched_u1_angles(Lx, Lt, 2.0, 2, 5))).to(DEV)
    x = torch.from_numpy(W.gaussian_field((nrhs, Lt, Lx, 2), 8)).to(torch.complex64).to(DEV)
    with mg.Multigrid(U, -1.9, [], [], autotune=0) as s:
        y, ref = torch.empty_like(x), torch.empty(x.shape, dtype=torch.complex128, device=DEV)
        mg.mg_apply_A(s.h, x, y, nrhs, mg.PREC_F32)
        mg.mg_apply_A(s.h, x.to(torch.complex128), ref, nrhs, mg.PREC_F64)
    big = torch.maximum(x.real.abs(), x.imag.abs()).amax(-1).double()
    loc = torch.stack([torch.roll(big, (dt, dx), (1, 2)) for dt in range(-2, 3)
                       for dx in range(-2 + abs(dt), 3 - abs(dt))]).amax(0)
    tol = 45 * 2.0 ** -24 * 6.1 ** 2 * loc[..., None]
    assert torch.all((y.to(torch.complex128) - ref).abs() <= tol)


def test_vcycle_epilogues(mg):
    """A batched mixed solve runs every epilogue of the streaming stencil (r = b - A x, x += R r)."""
    Lx, Lt, nrhs = 128, 128, 24
    U = torch.from_numpy(W.links_from_angles(W.quenched_u1_angles(Lx, Lt, 6.0, 5, 5))).to(DEV)
    noise = torch.from_numpy(W.setup_noise(Lx, Lt, [(4, 4), (2, 2)], [4, 4], 7)).to(DEV)
    b = torch.from_numpy(W.gaussian_field((nrhs, Lt, Lx, 2), 8)).to(DEV)
    with mg.Multigrid(U, -1.9, [(4, 4), (2, 2)], [4, 4], noise, autotune=0, max_rhs=nrhs) as s:
        _, batch = s.solve(b, tol=1e-10)
    with mg.Multigrid(U, -1.9, [(4, 4), (2, 2)], [4, 4], noise, autotune=0) as s:
        _, one = s.solve(b[:1].contiguous(), tol=1e-10)
    assert all(i.true_residual <= 1e-10 for i in batch)
    assert abs(batch[0].iterations - one[0].iterations) <= 1   # the same preconditioner in tiles
