"""The 2-d operator at the edges of its launch rules, against the oracle on the whole lattice: thread
counts on both sides of 152 x 256 (blocks of 64 and of 128), lattices whose last block is partial,
and slice walks of 1, 2, 4 and all slices whose last walk is shorter than the others."""
import numpy as np
import pytest
import torch

import synth
from oracle import dirac

pytestmark = pytest.mark.gpu

TOL = {"f64": 1e-12, "f32": 1e-5, "f32_l16": 1e-5}


@pytest.fixture(scope="module")
def dw():
    if not torch.cuda.is_available():
        pytest.skip("no GPU")
    import paper_2004_07732_gb300 as pkg
    pkg.lib()
    return pkg


# FP32 walks: 48 x 50 and 811 x 3 one slice (38,400 and 38,928 threads); 197 x 197 two; 281 x 139 four, then
# three; 283 x 275 all five.  FP64: one slice for the first four, two (the last walk one) for 283 x 275.
@pytest.mark.parametrize("dims,Ls,anti", [((48, 50), 16, None), ((811, 3), 16, [0, 1]), ((197, 197), 4, [1, 0]),
                                         ((281, 139), 7, None), ((283, 275), 5, [1, 1])])
@pytest.mark.parametrize("prec", ["f64", "f32", "f32_l16"])
def test_walks_and_blocks(dw, dims, Ls, anti, prec):
    rng = synth.rng_for(107)
    U = synth.u1_links(synth.u1_angles(rng, dims, 0.6))
    psi = synth.gaussian_spinor(rng, dims, Ls)
    if prec == "f32_l16":
        U = U.real.astype(np.float16).astype(np.float64) + 1j * U.imag.astype(np.float16).astype(np.float64)
    g = dw.make_geom(dims, Ls, antiperiodic=anti)
    Ud = dw.links_to(g, torch.from_numpy(np.ascontiguousarray(U).reshape(-1)).to("cuda"), prec)
    p = torch.from_numpy(psi.reshape(-1)).to("cuda").to(dw.spinor_dtype(prec))
    for dag in (False, True):
        out = dw.dwf_apply(g, Ud, p, torch.full_like(p, 5.0), 1.0, 0.05, dagger=dag, prec=prec).cpu().numpy()
        want = dirac.dwf_apply(U, psi, dims, Ls, 1.0, 0.05, dag, antiperiodic=anti).reshape(-1)
        assert np.linalg.norm(out - want) <= TOL[prec] * np.linalg.norm(want)
        # no site or slice left out: the largest single error, against the oracle's mean
        assert np.abs(out - want).max() <= 100 * TOL[prec] * np.abs(want).mean()
