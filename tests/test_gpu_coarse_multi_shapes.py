"""GPU parity of the many-right-hand-side coarse operator on FP16 blocks, one column tile at a time
(coarse_tc = 2), at the shapes where its kernel can go wrong: coarse extents of 1, 2 and ones that do not
fill a tile of 4 x 4 sites, column counts that do not fill a tile of 8 or share it between
right-hand sides, columns of very different size, zero columns, and both vector layouts.  The blocks are the library's own,
rounded to FP16; the sum is written out here.  Tolerance 1e-5 relative per column, as for the
other FP32 stencils."""
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


@pytest.mark.parametrize("cdims,Ls_c,nrhs", [((1, 3), 1, 5), ((2, 2), 4, 1), ((5, 3), 3, 7), ((9, 6), 4, 3),
                                             ((4, 8), 2, 20), ((6, 1), 8, 3)])
@pytest.mark.parametrize("layout", ["slice_major", "site_major"])
def test_multi_vector_shapes(dw, cdims, Ls_c, nrhs, layout):
    dims, nvec, mf = tuple(4 * c for c in cdims), 8, 0.07
    rng = synth.rng_for(107)
    U = synth.u1_links(synth.u1_angles(rng, dims, 0.5))
    V, Vc = int(np.prod(dims)), int(np.prod(cdims))
    starts = synth.gaussian_complex(rng, (nvec, V * 2))
    h = dw.mg_setup(dw.make_geom(dims, 8), _dev(U), 1.0, 0.05, {"setup_maxiter": 0, "Ls_c": Ls_c, "coarse_tc": 2},
                    _dev(starts))
    Y = dw.mg_get_coarse_links(h).cpu().numpy().reshape(Vc, 5, 16, 16)
    Y = Y.real.astype(np.float16).astype(float) + 1j * Y.imag.astype(np.float16).astype(float)
    x, y = np.arange(Vc) % cdims[0], np.arange(Vc) // cdims[0]
    nbs = [np.arange(Vc)]
    for sx, sy in ((1, 0), (-1, 0), (0, 1), (0, -1)):
        nbs.append((x + sx) % cdims[0] + (y + sy) % cdims[1] * cdims[0])
    v = synth.gaussian_complex(rng, (nrhs, Ls_c, Vc, 16))
    v *= 10.0 ** rng.uniform(-25, 25, (nrhs, 1, 1, 1))
    v[nrhs // 2, 0] = 0.0
    v = v.astype(np.complex64).astype(complex)
    order = (0, 1, 2, 3) if layout == "slice_major" else (2, 0, 1, 3)
    back = np.argsort(order)
    sig = np.where(np.arange(16) < 8, 1.0, -1.0)
    for dag in (False, True):
        s3 = sig if dag else np.ones(16)
        want = v + s3 * sum(np.einsum("xab,rsxb->rsxa", Y[:, d], (v * s3)[:, :, nbs[d]]) for d in range(5))
        for s in range(Ls_c):
            lo = (v[:, s - 1] if s > 0 else -mf * v[:, Ls_c - 1])
            hi = (v[:, s + 1] if s + 1 < Ls_c else -mf * v[:, 0])
            plus, minus = (hi, lo) if dag else (lo, hi)
            want[:, s, :, :8] += plus[..., :8]
            want[:, s, :, 8:] += minus[..., 8:]
        vin = _dev(v.transpose(order), torch.complex64)
        out = dw.mg_coarse_apply_multi(h, vin, torch.empty_like(vin), nrhs, mf, dag, layout=layout)
        got = out.cpu().numpy().reshape(np.array(v.shape)[list(order)]).transpose(back)
        for r in range(nrhs):
            for s in range(Ls_c):
                assert np.linalg.norm(got[r, s] - want[r, s]) <= 1e-5 * np.linalg.norm(want[r, s])
    h.close()
