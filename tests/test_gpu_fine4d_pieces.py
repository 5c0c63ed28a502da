"""The canonical 4-d operator on spinors that start on a 32-byte boundary (32-byte pieces) and on
ones that start 16 bytes past it (16-byte pieces): against the oracle, at the tolerances of the
other parity tests, and the same bits from both.  Lattices whose sites do not fill the last thread
block and whose slices do not fill the last group of eight."""
import numpy as np
import pytest
import torch

import synth
from oracle import dirac

pytestmark = pytest.mark.gpu


@pytest.fixture(scope="module")
def dw():
    if not torch.cuda.is_available():
        pytest.skip("no GPU")
    import paper_2004_07732_gb300 as pkg
    pkg.lib()
    return pkg


def _at(t, shift):
    """The values of t at 16 * shift bytes past a 32-byte boundary."""
    n = 16 * shift // t.element_size()
    room = torch.zeros(t.numel() + n, dtype=t.dtype, device=t.device)
    assert room.data_ptr() % 32 == 0
    room[n:].copy_(t)
    return room[n:]


@pytest.mark.parametrize("dims,Ls,anti", [((3, 2, 5, 2), 3, None), ((1, 4, 2, 3), 9, [1, 0, 0, 1])])
@pytest.mark.parametrize("prec,tol", [("f64", 1e-12), ("f32", 1e-5)])
def test_aligned_and_shifted_spinors(dw, dims, Ls, anti, prec, tol):
    rng = synth.rng_for(103)
    U = synth.su3_links(rng, dims, 0.4)
    psi = synth.gaussian_spinor(rng, dims, Ls, "su3")
    g = dw.make_geom(dims, Ls, "su3", anti)
    Ud = dw.links_to(g, torch.from_numpy(U.reshape(-1)).to("cuda"), prec)
    p = torch.from_numpy(psi.reshape(-1)).to("cuda").to(dw._lib.spinor_dtype(prec))
    for dag in (False, True):
        got = []
        for a, b in ((0, 0), (1, 1), (0, 1), (1, 0)):
            out = _at(torch.full_like(p, 5.0), b)
            got.append(dw.dwf_apply(g, Ud, _at(p, a), out, 1.8, 0.05, dag, prec).cpu().numpy())
        want = dirac.dwf_apply(U, psi, dims, Ls, 1.8, 0.05, dag, "su3", anti).reshape(-1)
        assert np.linalg.norm(got[0] - want) <= tol * np.linalg.norm(want)
        for other in got[1:]:
            assert np.array_equal(got[0], other)
