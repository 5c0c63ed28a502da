"""GPU parity of the 48-dof coarse operator (4-d SU(3), 24 vectors, FP16 blocks) at the shapes
where its kernel can go wrong: coarse extents of 1, 2 and odd ones (a neighbour may be the site
itself, or the same site in both directions), sites that do not fill the last thread block, 1 to 4
coarse slices, vectors that are only 8-byte aligned, and slices of very different size (each is
scaled by itself), zero ones among them.  The blocks are the library's own, rounded to FP16; the sum is written
out here.  Tolerance 1e-5 relative per slice, as for the other FP32 stencils."""
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


def _dev(a, dtype=torch.complex128):
    return torch.from_numpy(np.ascontiguousarray(a).reshape(-1)).to("cuda").to(dtype)


def _offset(t):
    """The same values at an address that is 8 and not 16 bytes aligned."""
    return torch.cat([torch.zeros(1, dtype=t.dtype, device=t.device), t])[1:]


@pytest.mark.parametrize("cdims,Ls_c,anti", [((1, 2, 3, 1), 4, None), ((2, 2, 2, 3), 3, [0, 0, 0, 1]),
                                             ((3, 1, 2, 2), 1, [1, 0, 1, 0]), ((2, 3, 1, 3), 2, None)])
def test_48dof_shapes(dw, cdims, Ls_c, anti):
    dims, nvec, mf = tuple(2 * c for c in cdims), 24, 0.07
    rng = synth.rng_for(101)
    U = synth.su3_links(rng, dims, 0.3)
    V, Vc = int(np.prod(dims)), int(np.prod(cdims))
    starts = synth.gaussian_complex(rng, (nvec, V * 12))
    h = dw.mg_setup(dw.make_geom(dims, 6, "su3", anti), _dev(U), 1.8, 0.05,
                    {"nvec": nvec, "block": [2, 2, 2, 2], "setup_maxiter": 0, "Ls_c": Ls_c}, _dev(starts))
    Y = dw.mg_get_coarse_links(h).cpu().numpy().reshape(Vc, 9, 48, 48)
    c = np.indices(tuple(reversed(cdims))).reshape(4, -1)[::-1]        # coordinate mu of every site
    nbs = [np.arange(Vc)]
    for mu in range(4):
        for step in (1, -1):
            d = c.copy()
            d[mu] = (d[mu] + step) % cdims[mu]
            nbs.append(d[0] + cdims[0] * (d[1] + cdims[1] * (d[2] + cdims[2] * d[3])))
    sig = np.where(np.arange(48) < 24, 1.0, -1.0)
    # the backward block of x is sigma_3 (forward block of x - mu)^dag sigma_3, exactly
    for mu in range(4):
        want = sig[:, None] * np.conj(np.swapaxes(Y[nbs[2 + 2 * mu], 1 + 2 * mu], -1, -2)) * sig
        assert np.array_equal(Y[:, 2 + 2 * mu], want)
    Y = Y.real.astype(np.float16).astype(float) + 1j * Y.imag.astype(np.float16).astype(float)
    v = synth.gaussian_complex(rng, (Ls_c, Vc, 48)) * np.array([1.0, 1e-30, 1e25, 0.0])[:Ls_c, None, None]
    v[0, Vc - 1] = 0.0
    v = v.astype(np.complex64).astype(complex)
    for dag in (False, True):
        s3 = sig if dag else np.ones(48)
        hop = s3 * sum(np.einsum("xab,sxb->sxa", Y[:, d], (v * s3)[:, nbs[d]]) for d in range(9)) + v
        want = hop.copy()
        for s in range(Ls_c):
            lo = (v[s - 1] if s > 0 else -mf * v[Ls_c - 1])
            hi = (v[s + 1] if s + 1 < Ls_c else -mf * v[0])
            plus, minus = (hi, lo) if dag else (lo, hi)
            want[s, :, :24] += plus[:, :24]
            want[s, :, 24:] += minus[:, 24:]
        for move in (lambda t: t, _offset):
            out = move(torch.empty(v.size, dtype=torch.complex64, device="cuda"))
            got = dw.mg_coarse_apply(h, move(_dev(v, torch.complex64)), out, mf, dag).cpu().numpy().reshape(v.shape)
            for s in range(Ls_c):
                assert np.linalg.norm(got[s] - want[s]) <= 1e-5 * np.linalg.norm(want[s])
    h.close()
