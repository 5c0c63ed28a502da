"""The bulk prolongation (one coarse slice onto each fine one) where a thread takes one slice and where
it takes several, not the same number each: against the sum over the library's own prolongator.
Tolerance: FP32 sums of nvec products, 1e-6 relative (nvec 2^-24 = 1.8e-7 at most)."""
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


# 240 blocks of (site, chirality) threads: two of the three slices to one; 640: all three; 32: one each
@pytest.mark.parametrize("dims", [(192, 160), (256, 320), (64, 64)])
def test_bulk_prolongation(dw, dims):
    Ls, nvec = 3, 3
    rng = synth.rng_for(191)
    V = dims[0] * dims[1]
    U = synth.u1_links(synth.u1_angles(rng, dims, 0.5))
    starts = torch.from_numpy(synth.gaussian_complex(rng, (nvec * V * 2,))).to("cuda")
    h = dw.mg_setup(dw.make_geom(dims, Ls), torch.from_numpy(U.reshape(-1)).to("cuda"), 1.0, 0.05,
                    {"nvec": nvec, "block": [4, 4], "Ls_c": Ls, "transfer": 1, "setup_maxiter": 0}, starts)
    P = dw.mg_get_prolongator(h).reshape(V, 2, nvec)
    e = torch.from_numpy(synth.gaussian_complex(rng, (Ls, V // 16, 2, nvec)).astype(np.complex64)).to("cuda")
    got = dw.mg_prolong(h, e.reshape(-1), torch.full((Ls * V * 2,), 7.0, dtype=torch.complex64, device="cuda"))
    x, y = torch.arange(V, device="cuda") % dims[0], torch.arange(V, device="cuda") // dims[0]
    want = (P[None] * e[:, y // 4 * (dims[0] // 4) + x // 4]).sum(-1)
    assert float((got.reshape(want.shape) - want).norm()) <= 1e-6 * float(want.norm())
    h.close()
