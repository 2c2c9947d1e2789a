"""FP32 restriction and prolongation at the edges of the register kernels: lattices whose rows end
inside a warp, every supported number of vectors and one that is not, chunks of right-hand sides
with remainders, and coarse vectors that are only 8-byte aligned, against the FP64 kernels.

Tolerance: a sum of T products in FP32 with FP32 block vectors is off by at most (T + 3) 2^-24 of
the sum of magnitudes; with orthonormal vectors that sum is at most the norm of the block's input
(restriction, T = bx bt h) or of the site's coarse input (prolongation, T = Nv)."""
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


def _apply(mg, f, h, level, x, shape, prec, shift=0):
    dt = torch.complex128 if prec == mg.PREC_F64 else torch.complex64
    buf = torch.empty(x.size + shift, dtype=dt, device=DEV)
    xt = buf[shift:].view(x.shape)
    xt.copy_(torch.from_numpy(x).to(DEV))
    out = torch.empty(int(np.prod(shape)) + shift, dtype=dt, device=DEV)[shift:].view(shape)
    f(h, level, xt, out, x.shape[0], prec)
    return out.cpu().numpy()


@pytest.mark.parametrize("Lx,Lt,Nv,nrhs,shift", [
    (16, 16, 4, 1, 0), (24, 16, 8, 3, 0), (40, 24, 8, 64, 0), (24, 16, 12, 5, 0), (72, 16, 12, 1, 0), (24, 16, 6, 2, 0),
    (24, 16, 8, 3, 1)])
def test_transfers(mg, Lx, Lt, Nv, nrhs, shift):
    U = torch.from_numpy(W.links_from_angles(W.quenched_u1_angles(Lx, Lt, 3.0, 2, 5))).to(DEV)
    blocks = [(4, 4), (2, 2)]
    noise = torch.from_numpy(W.setup_noise(Lx, Lt, blocks, [Nv, Nv], 7)).to(DEV)
    with mg.Multigrid(U, -1.9, blocks, [Nv, Nv], noise, autotune=0) as s:
        for level, (bx, bt), n in ((1, (4, 4), 2), (2, (2, 2), 2 * Nv)):
            lx, lt = Lx // (1 if level == 1 else 4), Lt // (1 if level == 1 else 4)
            fs, cs = (nrhs, lt, lx, n), (nrhs, lt // bt, lx // bx, 2 * Nv)
            f = W.gaussian_field(fs, 3).astype(np.complex64).astype(np.complex128)
            e = W.gaussian_field(cs, 4).astype(np.complex64).astype(np.complex128)
            r = {p: _apply(mg, mg.mg_restrict, s.h, level, f, cs, p, shift) for p in (mg.PREC_F64, mg.PREC_F32)}
            blk = f.reshape(nrhs, lt // bt, bt, lx // bx, bx, 2, n // 2)
            norm = np.sqrt((np.abs(blk) ** 2).sum((2, 4, 6)))                 # [rhs][jt][jx][chirality]
            tol = (bx * bt * n // 2 + 3) * 2.0 ** -24 * np.repeat(norm, Nv, -1)
            assert np.all(np.abs(r[mg.PREC_F32] - r[mg.PREC_F64]) <= tol), level
            p = {q: _apply(mg, mg.mg_prolong, s.h, level, e, fs, q, shift) for q in (mg.PREC_F64, mg.PREC_F32)}
            norm = np.sqrt((np.abs(e.reshape(cs[:3] + (2, Nv))) ** 2).sum(-1))
            tol = (Nv + 3) * 2.0 ** -24 * np.repeat(np.repeat(norm, bt, 1), bx, 2)
            assert np.all(np.abs(p[mg.PREC_F32] - p[mg.PREC_F64]) <= np.repeat(tol, n // 2, -1)), level
