"""The FP32 streaming stencil keeps the range of its results: a field whose A psi reaches between a
quarter and a half of the largest FP32 number gives exactly the scaled result of the field at
order one (a power of two apart), in tiles and streamed.  And the accuracy of test_gpu_stencil_stream at
sizes large enough to be streamed whose last strip of 60 sites is full, one pair and half wide."""
import math

import numpy as np
import pytest

import workloads as W
from test_gpu_stencil_stream import mg, test_streaming_stencil as _accuracy  # noqa: F401

torch = pytest.importorskip("torch")
pytestmark = pytest.mark.gpu

DEV = "cuda:0"


@pytest.mark.parametrize("Lx,Lt,nrhs", [(32, 32, 1), (256, 250, 33), (1024, 256, 4)])
def test_large_results(mg, Lx, Lt, nrhs):  # noqa: F811
    U = torch.from_numpy(W.links_from_angles(W.quenched_u1_angles(Lx, Lt, 2.0, 2, 5))).to(DEV)
    x = torch.from_numpy(W.gaussian_field((nrhs, Lt, Lx, 2), 8)).to(torch.complex64).to(DEV)
    with mg.Multigrid(U, -1.9, [], [], autotune=0) as s:
        y, z = torch.empty_like(x), torch.empty_like(x)
        mg.mg_apply_A(s.h, x, y, nrhs, mg.PREC_F32)
        top = torch.view_as_real(y).abs().max().item()
        scale = 2.0 ** (127 - math.frexp(top)[1])            # the largest in [2^126, 2^127)
        mg.mg_apply_A(s.h, x * scale, z, nrhs, mg.PREC_F32)
    a, b = torch.view_as_real(y).cpu().numpy(), torch.view_as_real(z).cpu().numpy()
    assert np.array_equal(a * np.float32(scale), b)


@pytest.mark.parametrize("Lx,Lt,nrhs", [(120, 250, 40), (122, 250, 30), (90, 130, 64)])
def test_last_strips(mg, Lx, Lt, nrhs):  # noqa: F811
    _accuracy(mg, Lx, Lt, nrhs)
