"""Rounding of the FP32 transfers against the FP64 ones on the same inputs.  An output is a
sum of products formed in chains that are added pairwise; the roundings of a chain of n
fused multiply-adds weigh (n + 1) / 2 of a rounding of the result in the mean square, every
level of pairwise additions one, and the rounding of the vectors to FP32 one.  Prolongation:
four chains of Nv / 2, two levels; restriction on 4 x 4 blocks: chains of 4, three levels.
One rounding is at most 2^-24 / sqrt(3) in the root mean square."""
import math

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


@pytest.mark.parametrize("nrhs", [1, 5])
@pytest.mark.parametrize("Nv", [4, 8, 12])
def test_rounding(mg, Nv, nrhs):
    Lx, Lt = 64, 48
    U = torch.from_numpy(W.quenched_u1(Lx, Lt, 6.0, 20, 3)).to(DEV)
    noise = torch.from_numpy(W.setup_noise(Lx, Lt, [(4, 4)], [Nv], 5)).to(DEV)
    g = torch.Generator(device=DEV).manual_seed(7)
    f = torch.randn((nrhs, Lt, Lx, 2), generator=g, device=DEV, dtype=torch.complex64)
    c = torch.randn((nrhs, Lt // 4, Lx // 4, 2 * Nv), generator=g, device=DEV, dtype=torch.complex64)
    f64, c64 = f.to(torch.complex128), c.to(torch.complex128)
    out = [torch.empty_like(t) for t in (c, f, c64, f64)]
    with mg.Multigrid(U, 0.0, [(4, 4)], [Nv], noise) as s:
        mg.mg_restrict(s.h, 1, f, out[0], nrhs, mg.PREC_F32)
        mg.mg_prolong(s.h, 1, c, out[1], nrhs, mg.PREC_F32)
        mg.mg_restrict(s.h, 1, f64, out[2], nrhs, mg.PREC_F64)
        mg.mg_prolong(s.h, 1, c64, out[3], nrhs, mg.PREC_F64)
        torch.cuda.synchronize()
    for got, want, n in ((out[0], out[2], 2.5 + 3 + 1), (out[1], out[3], (Nv / 2 + 1) / 2 + 2 + 1)):
        err = torch.linalg.vector_norm(got - want) / torch.linalg.vector_norm(want)
        assert err.item() <= math.sqrt(n / 3) * 2 ** -24
