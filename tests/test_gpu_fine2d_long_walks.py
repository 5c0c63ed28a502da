"""GPU parity of the 2-d operator in FP32 on more than 16 slices, where the length of a thread's walk
along s follows from the rounds of thread blocks: in one round of 921 blocks (14 slices each), in
between (1250 and more blocks: 16 slices and a rest), and from four rounds on (the whole of s).
Tolerance 1e-6 relative: each value is a sum of about 20 FP32 products."""
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


@pytest.mark.parametrize("dims,Ls,anti", [((200, 196), 40, [1, 0]), ((398, 403), 33, None), ((790, 789), 17, [0, 1])])
def test_long_walks(dw, dims, Ls, anti):
    rng = synth.rng_for(139)
    U = synth.u1_links(synth.u1_angles(rng, dims, 0.6))
    psi = synth.gaussian_spinor(rng, dims, Ls)
    g = dw.make_geom(dims, Ls, antiperiodic=anti)
    Ud = dw.links_to(g, torch.from_numpy(U.reshape(-1)).to("cuda"), "f32")
    p = torch.from_numpy(psi.reshape(-1)).to("cuda").to(torch.complex64)
    for dag in (False, True):
        out = dw.dwf_apply(g, Ud, p, torch.full_like(p, 5.0), 1.0, 0.05, dagger=dag, prec="f32").cpu().numpy()
        want = dirac.dwf_apply(U, psi, dims, Ls, 1.0, 0.05, dag, antiperiodic=anti).reshape(-1)
        assert np.linalg.norm(out - want) <= 1e-6 * np.linalg.norm(want)
        # no site or slice left out: the largest single error, against the oracle's mean
        assert np.abs(out - want).max() <= 1e-4 * np.abs(want).mean()
