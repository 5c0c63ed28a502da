"""GPU parity of the one-vector coarse operator (2-d, 16 coarse dof) at the shapes where its
kernel can go wrong: coarse extents of 1, 2 and odd ones (a neighbour may be the site itself), a
number of sites that does not fill the last thread block, 1 to 4 coarse slices, FP16 and FP32 blocks,
and vectors that are only 8-byte aligned.  The blocks are the library's own (rounded to FP16 where
it stores them so); the sum is written out here.  1e-5 relative, as for the other FP32 stencils."""
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


@pytest.mark.parametrize("cdims,Ls_c", [((1, 3), 1), ((2, 2), 2), ((5, 3), 3), ((7, 4), 4), ((3, 1), 4)])
@pytest.mark.parametrize("prec", ["f32", "f32_l16"])
@pytest.mark.parametrize("shift", [False, True])
def test_one_vector_shapes(dw, cdims, Ls_c, prec, shift):
    dims, nvec, mf = tuple(4 * c for c in cdims), 8, 0.07
    rng = synth.rng_for(97)
    U = synth.u1_links(synth.u1_angles(rng, dims, 0.5))
    V, Vc = int(np.prod(dims)), int(np.prod(cdims))
    starts = synth.gaussian_complex(rng, (nvec, V * 2))
    h = dw.mg_setup(dw.make_geom(dims, 6), _dev(U), 1.0, 0.05,
                    {"setup_maxiter": 0, "Ls_c": Ls_c, "coarse_block_prec": prec}, _dev(starts))
    Y = dw.mg_get_coarse_links(h).cpu().numpy().reshape(Vc, 5, 16, 16)
    rnd = np.float16 if prec == "f32_l16" else np.float32
    Y = Y.real.astype(rnd).astype(float) + 1j * Y.imag.astype(rnd).astype(float)
    x, y = np.arange(Vc) % cdims[0], np.arange(Vc) // cdims[0]
    nbs = [np.arange(Vc)]
    for sx, sy in ((1, 0), (-1, 0), (0, 1), (0, -1)):
        nbs.append((x + sx) % cdims[0] + (y + sy) % cdims[1] * cdims[0])
    v = synth.gaussian_complex(rng, (Ls_c, Vc, 16))
    sig = np.where(np.arange(16) < 8, 1.0, -1.0)
    move = _offset if shift else (lambda t: t)
    vin = move(_dev(v, torch.complex64))
    for dag in (False, True):
        s3 = sig if dag else np.ones(16)
        want = v + s3 * sum(np.einsum("xab,sxb->sxa", Y[:, d], (v * s3)[:, nbs[d]]) for d in range(5))
        for s in range(Ls_c):
            lo = (v[s - 1] if s > 0 else -mf * v[Ls_c - 1])
            hi = (v[s + 1] if s + 1 < Ls_c else -mf * v[0])
            plus, minus = (hi, lo) if dag else (lo, hi)
            want[s, :, :8] += plus[:, :8]
            want[s, :, 8:] += minus[:, 8:]
        out = move(torch.empty(v.size, dtype=torch.complex64, device="cuda"))
        got = dw.mg_coarse_apply(h, vin, out, mf, dag).cpu().numpy().reshape(v.shape)
        assert np.linalg.norm(got - want) <= 1e-5 * np.linalg.norm(want)
    h.close()
