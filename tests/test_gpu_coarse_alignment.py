"""The coarse operator on complex64 vectors that start on an 8-byte but not on a 16-byte boundary
(a view into a larger buffer), for every stencil: the answer is that of an aligned copy."""
import numpy as np
import pytest
import torch

import synth

pytestmark = pytest.mark.gpu


@pytest.fixture(scope="module")
def dw():
    if not torch.cuda.is_available():
        pytest.skip("no GPU")
    import paper_2004_07732_gb300 as pkg
    pkg.lib()
    return pkg


def _dev(a):
    return torch.from_numpy(np.ascontiguousarray(a).reshape(-1)).to("cuda")


@pytest.mark.parametrize("group,dims,params", [
    ("su3", (4, 4, 4, 4), {"nvec": 8}), ("su3", (4, 4, 4, 4), {"nvec": 8, "Ls_c": 6}), ("su3", (4, 4, 4, 4), {"nvec": 4}),
    ("su3", (4, 4, 4, 4), {"nvec": 12}), ("su3", (4, 4, 4, 4), {"nvec": 24}), ("u1", (8, 12), {"nvec": 8}),
    ("u1", (8, 12), {"nvec": 3})])
def test_vectors_on_an_8_byte_boundary(dw, group, dims, params):
    rng = synth.rng_for(181)
    V = int(np.prod(dims))
    if group == "u1":
        U, dof, M5 = synth.u1_links(synth.u1_angles(rng, dims, 0.4)), 2, 1.0
    else:
        U, dof, M5 = synth.su3_links(rng, dims, 0.3), 12, 1.8
        params = {**params, "block": [2, 2, 2, 2]}
    starts = synth.gaussian_complex(rng, (params["nvec"], V * dof))
    h = dw.mg_setup(dw.make_geom(dims, 6, group), _dev(U), M5, 0.05,
                    {"setup_mass": -0.1, "setup_maxiter": 10, **params}, _dev(starts))
    n = h.coarse_size
    room = torch.from_numpy(synth.gaussian_complex(rng, (n + 1,)).astype(np.complex64)).to("cuda")
    view, out = room[1:], torch.empty_like(room)[1:]
    assert view.data_ptr() % 16 == 8 and out.data_ptr() % 16 == 8
    for dagger in (False, True):
        dw.mg_coarse_apply(h, view, out, 0.05, dagger)
        want = dw.mg_coarse_apply(h, view.clone(), torch.empty(n, dtype=room.dtype, device="cuda"), 0.05, dagger)
        # sums of up to 9 x 48 FP32 products in another order: 2^-24 sqrt(432) = 1.2e-6 of their norm
        assert float((out - want).norm()) <= 2e-6 * float(want.norm())
    h.close()
