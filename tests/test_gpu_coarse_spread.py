"""The coarse operators that multiply FP16 parts of FP32 inputs, on inputs of very different size
within one coarse site.  The near-null vectors are single fine components, so that a coarse dof is
one component of a fine site and an output row depends on few inputs; the rows looked at do not see the large ones,
and have to be as accurate, relative to themselves, as if those were not there.

A pair of parts keeps 22 bits of every input; a row sums about 30 products in FP32.  Tolerance
1e-6 relative in norm over the rows looked at: 4 ulp of FP32."""
import numpy as np
import pytest
import torch

import synth

pytestmark = pytest.mark.gpu
TOL = 1e-6


@pytest.fixture(scope="module")
def dw():
    if not torch.cuda.is_available():
        pytest.skip("no GPU")
    import paper_2004_07732_gb300 as pkg
    pkg.lib()
    return pkg


def _dev(a, dtype=torch.complex128):
    return torch.from_numpy(np.ascontiguousarray(a).reshape(-1)).to("cuda").to(dtype)


def _coords(dims):
    """coordinate mu of every site, x0 fastest"""
    return np.indices(tuple(reversed(dims))).reshape(len(dims), -1)[::-1]


def _neighbours(cdims):
    """self, +mu, -mu for every direction"""
    c, stride = _coords(cdims), np.cumprod([1] + list(cdims))[:-1]
    out = [np.arange(c.shape[1])]
    for mu in range(len(cdims)):
        for step in (1, -1):
            d = c.copy()
            d[mu] = (d[mu] + step) % cdims[mu]
            out.append((d * stride[:, None]).sum(0))
    return out


def _apply(Y, v, nbs, mf, dag):
    """v: [...][s][site][dof], dof the two chiralities"""
    half = v.shape[-1] // 2
    s3 = np.where(np.arange(2 * half) < half, 1.0, -1.0) if dag else np.ones(2 * half)
    out = v + s3 * sum(np.einsum("xab,...xb->...xa", Y[:, d], (v * s3)[..., nb, :]) for d, nb in enumerate(nbs))
    below = np.concatenate([-mf * v[..., -1:, :, :], v[..., :-1, :, :]], -3)
    above = np.concatenate([v[..., 1:, :, :], -mf * v[..., :1, :, :]], -3)
    plus, minus = (above, below) if dag else (below, above)
    out[..., :half] += plus[..., :half]
    out[..., half:] += minus[..., half:]
    return out


def _round16(Y):
    return Y.real.astype(np.float16).astype(float) + 1j * Y.imag.astype(np.float16).astype(float)


def _spread(v, kind, large, small):
    """large: coarse dof (chirality +) at full size; the other dof small, "within": of all chiralities
    alike, "chirality": only those of chirality -, the others zero"""
    half = v.shape[-1] // 2
    size = np.full(2 * half, small)
    if kind == "chirality":
        size[:half] = 0.0
    size[large] = 1.0
    return (v * size).astype(np.complex64).astype(complex)


# 2^-27: an input in the range that both parts hold in full; 2^-45: a chirality of its own scale
@pytest.mark.parametrize("kind,small", [("within", 2.0 ** -27), ("chirality", 2.0 ** -45)])
def test_48dof_spread(dw, kind, small):
    cdims, Ls_c, nvec, mf = (2, 3, 2, 2), 4, 24, 0.07
    dims = tuple(2 * c for c in cdims)
    rng = synth.rng_for(127)
    U = synth.su3_links(rng, dims, 0.3)
    V, Vc = int(np.prod(dims)), int(np.prod(cdims))
    # vector k: component k % 6 of both chiralities on the site (x0, x1, 0, 0) = k // 6 of every aggregate
    x = _coords(dims) % 2
    place = np.where((x[2] == 0) & (x[3] == 0), x[0] + 2 * x[1], -1)
    starts = np.zeros((nvec, V, 2, 6), complex)
    for k in range(nvec):
        starts[k, place == k // 6, :, k % 6] = 1.0
    h = dw.mg_setup(dw.make_geom(dims, 6, "su3"), _dev(U), 1.8, 0.05,
                    {"nvec": nvec, "block": [2, 2, 2, 2], "setup_maxiter": 0, "Ls_c": Ls_c}, _dev(starts))
    Y = _round16(dw.mg_get_coarse_links(h).cpu().numpy().reshape(Vc, 9, 48, 48))
    rows = np.r_[0:6, 24:30]                             # site (0, 0): its neighbours are (1, 0) and (0, 1)
    large = np.arange(18, 24)                            # site (1, 1)
    assert not Y[:, :, rows][..., large].any() and Y[:, :, rows].any()
    v = _spread(synth.gaussian_complex(rng, (Ls_c, Vc, 48)), kind, large, small)
    for dag in (False, True):
        want = _apply(Y, v, _neighbours(cdims), mf, dag)[..., rows]
        vin = _dev(v, torch.complex64)
        got = dw.mg_coarse_apply(h, vin, torch.empty_like(vin), mf, dag).cpu().numpy().reshape(v.shape)[..., rows]
        assert np.linalg.norm(want) > 0
        assert np.linalg.norm(got - want) <= TOL * np.linalg.norm(want), (kind, dag)
    h.close()


@pytest.mark.parametrize("kind,small", [("within", 2.0 ** -27), ("chirality", 2.0 ** -45)])
def test_multi_vector_spread(dw, kind, small):
    """coarse_tc = 2: the many-vector operator on FP16 blocks, one column tile at a time"""
    cdims, Ls_c, nvec, nrhs, mf = (5, 3), 3, 8, 5, 0.07
    dims = tuple(4 * c for c in cdims)
    rng = synth.rng_for(131)
    U = synth.u1_links(synth.u1_angles(rng, dims, 0.5))
    V, Vc = int(np.prod(dims)), int(np.prod(cdims))
    # vector k: both components of the site (x0, x1) = (k % 4, k // 4) of every aggregate
    x = _coords(dims) % 4
    place = x[0] + 4 * x[1]
    starts = np.zeros((nvec, V, 2), complex)
    for k in range(nvec):
        starts[k, place == k] = 1.0
    h = dw.mg_setup(dw.make_geom(dims, 8), _dev(U), 1.0, 0.05, {"setup_maxiter": 0, "Ls_c": Ls_c, "coarse_tc": 2},
                    _dev(starts))
    Y = _round16(dw.mg_get_coarse_links(h).cpu().numpy().reshape(Vc, 5, 16, 16))
    rows = np.r_[0:2, 8:10]                              # sites (0, 0) and (1, 0)
    large = np.array([6])                                # site (2, 1)
    assert not Y[:, :, rows][..., large].any() and Y[:, :, rows].any()
    v = _spread(synth.gaussian_complex(rng, (nrhs, Ls_c, Vc, 16)), kind, large, small)
    for dag in (False, True):
        want = _apply(Y, v, _neighbours(cdims), mf, dag)[..., rows]
        vin = _dev(v, torch.complex64)
        got = dw.mg_coarse_apply_multi(h, vin, torch.empty_like(vin), nrhs, mf, dag).cpu().numpy()
        got = got.reshape(v.shape)[..., rows]
        for r in range(nrhs):
            assert np.linalg.norm(want[r]) > 0
            assert np.linalg.norm(got[r] - want[r]) <= TOL * np.linalg.norm(want[r]), (kind, dag, r)
    h.close()
