"""Sums of the link gradient over s: one slice of size 1 and others whose products are each below half
a unit in the last place of the whole sum.  Added one by one to it they would all be lost; summed
by themselves first (four slices of SU(3), one of U(1)) they are kept, but for those that share the
first slice's partial sum."""
import pytest
import torch

pytestmark = pytest.mark.gpu
LS = 12


@pytest.fixture(scope="module")
def dw():
    if not torch.cuda.is_available():
        pytest.skip("no GPU")
    import paper_2004_07732_gb300 as pkg
    pkg.lib()
    return pkg


# one thread per link over all slices (the larger lattice of each group), and slices split over threads
@pytest.mark.parametrize("dims,group", [((16, 16, 16, 10), "su3"), ((6, 4, 4, 6), "su3"), ((400, 400), "u1"),
                                        ((32, 20), "u1")])
def test_small_slices_count(dw, dims, group):
    g = dw.make_geom(dims, LS, group)
    V = 1
    for n in dims:
        V *= n
    spins, colors, terms = (4, 3, 8) if group == "su3" else (2, 1, 4)   # products per slice and real number
    # upper spins 1 + i, lower ones 0: every product of the real part is the same
    x = torch.zeros(LS, V, spins, colors, dtype=torch.complex128, device="cuda")
    x[:, :, :spins // 2] = 1 + 1j
    lam = x.clone()
    small = terms * 2.0 ** -54                                         # a quarter of a unit in the last place of `terms`
    lam[1:] *= small
    grad = dw.link_grad(g, lam.reshape(-1), x.reshape(-1)).real
    want = -0.5 * (terms + (LS - 1) * terms * small)
    # what the slices that share the first one's sum may lose: `terms` products each
    shared = 3 if group == "su3" else 0
    assert float((grad - want).abs().max()) <= 0.5 * shared * terms * small
