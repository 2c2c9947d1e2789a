"""A chain of dependent launches gives the bits of the same chain in a captured graph, where
every kernel is launched plainly after its predecessor: one V-cycle (stencils, transfers, coarse
applies, the coarsest product) over many fresh inputs, in both precisions."""
import numpy as np
import pytest

import workloads as W

torch = pytest.importorskip("torch")
pytestmark = pytest.mark.gpu

DEV = "cuda:0"


@pytest.mark.parametrize("precision", ["f32", "f64"])
def test_dependent_and_plain_launches_agree(precision):
    if not torch.cuda.is_available():
        pytest.skip("no CUDA device")
    import __graft_entry__
    __graft_entry__.build()
    from paper_0710_3612_gb300 import mg
    Lx, Lt, blocks, Nv = 64, 48, [(4, 4), (2, 2)], [8, 8]
    prec, dt = (mg.PREC_F32, torch.complex64) if precision == "f32" else (mg.PREC_F64, torch.complex128)
    U = W.links_from_angles(W.quenched_u1_angles(Lx, Lt, 6.0, 10, 1))
    noise = W.setup_noise(Lx, Lt, blocks, Nv, 7)
    stream = torch.cuda.Stream()
    with torch.cuda.stream(stream):
        with mg.Multigrid(torch.from_numpy(U).to(DEV), -0.2, blocks, Nv, torch.from_numpy(noise).to(DEV)) as s:
            x = torch.empty((Lt, Lx, 2), dtype=dt, device=DEV)
            eager, plain = torch.empty_like(x), torch.empty_like(x)
            mg.mg_vcycle(s.h, x.zero_(), eager, prec)
            stream.synchronize()
            graph = torch.cuda.CUDAGraph()
            with torch.cuda.graph(graph, stream=stream):
                mg.mg_vcycle(s.h, x, plain, prec)
            gen = torch.Generator(device=DEV)
            gen.manual_seed(3)
            for _ in range(300):
                x.copy_(torch.view_as_complex(torch.randn((Lt, Lx, 2, 2), generator=gen, device=DEV)))
                mg.mg_vcycle(s.h, x, eager, prec)
                graph.replay()
                assert torch.equal(torch.view_as_real(eager), torch.view_as_real(plain))
            assert np.isfinite(torch.linalg.vector_norm(plain).item())
