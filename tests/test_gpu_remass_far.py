"""A re-mass far from the set-up mass keeps the coarse operators as accurate as Galerkin products at
the new mass: the mass coefficients (remass_quadratic) against the products, by set_mass and by
clone, there and back.  Both sides add up to 72 rounded products per entry (8 units of 2^-53 of the
largest entry at random, twice) and the combination costs three bits at most on three terms:
40 units of 2^-52."""
import pytest

import workloads as W

torch = pytest.importorskip("torch")
pytestmark = pytest.mark.gpu

DEV = "cuda:0"
LX, LT, BLOCKS, NV = 32, 32, [(4, 4), (2, 2)], [4, 4]


@pytest.fixture(scope="module")
def mg():
    if not torch.cuda.is_available():
        pytest.skip("no CUDA device")
    import __graft_entry__
    __graft_entry__.build()
    from paper_0710_3612_gb300 import mg as m
    return m


def _ops(mg, h):
    out, lt, lx = [], LT, LX
    for l, ((bx, bt), nv) in enumerate(zip(BLOCKS, NV)):
        lx, lt = lx // bx, lt // bt
        out.append(torch.empty((lt, lx, 9, 2 * nv, 2 * nv), dtype=torch.complex128, device=DEV))
        mg.mg_get_coarse_op(h, l + 2, out[-1])
    return out


@pytest.mark.parametrize("masses", [(60.0, -0.05), (30.0, -1.5, 30.0), (-1.5, 60.0, -0.05), (0.1, -1.5), (5.0, 1.0, -1.5)])
def test_operators(mg, masses):
    U = torch.from_numpy(W.links_from_angles(W.quenched_u1_angles(LX, LT, 6.0, 10, 1))).to(DEV)
    noise = torch.from_numpy(W.setup_noise(LX, LT, BLOCKS, NV, 7)).to(DEV)
    with mg.Multigrid(U, masses[0], BLOCKS, NV, noise) as quad, \
            mg.Multigrid(U, masses[0], BLOCKS, NV, noise, remass_quadratic=0) as product:
        for m in masses[1:]:
            clone = mg.mg_clone(quad.h, m)
            quad.set_mass(m)
            product.set_mass(m)
            want = _ops(mg, product.h)
            for h in (quad.h, clone):
                for a, b in zip(_ops(mg, h), want):
                    assert (a - b).abs().max() <= 40 * 2.0 ** -52 * b.abs().max(), m
            mg.mg_destroy(clone)
