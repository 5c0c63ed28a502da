"""GPU parity of the wall and bulk transfers at the sizes where their kernels change course:
odd and even numbers of vectors (8- and 16-byte accesses), vectors that are only 8-byte aligned,
one and two slices, aggregates too large for the offset table, and the packed 4-d layout with
two, four and more slices.  The prolongator is the library's own; the sums are written out here.
Tolerance: FP32 sums of at most nb * nchd terms, 1e-5 relative as in the other FP32 parity tests."""
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


def _setup(dw, dims, block, nvec, Ls, Ls_c, extra=None):
    rng = synth.rng_for(83)
    group = "u1" if len(dims) == 2 else "su3"
    U = synth.u1_links(synth.u1_angles(rng, dims, 0.5)) if group == "u1" else synth.su3_links(rng, dims, 0.3)
    V, dof = int(np.prod(dims)), 2 if group == "u1" else 12
    starts = synth.gaussian_complex(rng, (nvec, V * dof))
    g = dw.make_geom(dims, Ls, group)
    prm = {"nvec": nvec, "block": list(block), "Ls_c": Ls_c, "setup_maxiter": 0, **(extra or {})}
    return dw.mg_setup(g, _dev(U), 1.0, 0.05, prm, _dev(starts)), rng, V, dof


def _aggregates(dims, block):
    """[coarse site][site of it]: fine site indices, x0 fastest in both."""
    c = np.indices(tuple(reversed(dims))).reshape(len(dims), -1)[::-1]        # coordinate mu of every site
    agg, stride = 0, 1
    for mu, (L, b) in enumerate(zip(dims, block)):
        agg = agg + c[mu] // b * stride
        stride *= L // b
    order = np.argsort(agg, kind="stable")
    return order.reshape(stride, -1)


@pytest.mark.parametrize("dims,block,nvec,Ls,Ls_c,bulk", [
    ((8, 12), (4, 4), 8, 6, 4, 0), ((8, 12), (4, 3), 3, 5, 1, 0), ((12, 8), (2, 4), 1, 2, 2, 0),
    ((8, 8), (2, 2), 2, 1, 1, 0), ((8, 8), (2, 2), 3, 3, 3, 1), ((128, 64), (64, 64), 2, 3, 2, 0),
    ((4, 2, 4, 6), (2, 2, 2, 2), 6, 4, 3, 0), ((4, 4, 2, 4), (2, 2, 1, 2), 5, 2, 2, 1)])
@pytest.mark.parametrize("shift", [False, True])
def test_transfer_shapes(dw, dims, block, nvec, Ls, Ls_c, bulk, shift):
    h, rng, V, dof = _setup(dw, dims, block, nvec, Ls, Ls_c, {"transfer": bulk})
    P = dw.mg_get_prolongator(h).cpu().numpy().reshape(V, 2, dof // 2, nvec)
    agg = _aggregates(dims, block)
    Vc = len(agg)
    r = synth.gaussian_complex(rng, (Ls, V, 2, dof // 2))
    e = synth.gaussian_complex(rng, (Ls_c, Vc, 2, nvec))
    rc = np.zeros((Ls_c, Vc, 2, nvec), complex)
    ef = np.zeros((Ls, V, 2, dof // 2), complex)
    walls = [(s, s, c) for s in range(Ls) for c in (0, 1)] if bulk else [(0, 0, 1), (Ls - 1, Ls_c - 1, 0)]
    for s, sc, c in walls:
        for a, sites in enumerate(agg):
            rc[sc, a, c] = np.einsum("xdk,xd->k", np.conj(P[sites, c]), r[s, sites, c])
            ef[s, sites, c] = np.einsum("xdk,k->xd", P[sites, c], e[sc, a, c])
    move = _offset if shift else (lambda t: t)
    got_r = dw.mg_restrict(h, move(_dev(r, torch.complex64)), move(torch.empty(rc.size, dtype=torch.complex64,
                                                                               device="cuda")))
    out = move(torch.full((ef.size,), 7.0, dtype=torch.complex64, device="cuda"))
    got_e = dw.mg_prolong(h, move(_dev(e, torch.complex64)), out)
    for got, want in ((got_r, rc), (got_e, ef)):
        got = got.cpu().numpy().reshape(want.shape)
        assert np.linalg.norm(got - want) <= 1e-5 * np.linalg.norm(want)
        assert np.all(got[want == 0] == 0)
    h.close()


@pytest.mark.parametrize("Ls", [2, 4, 8])
def test_packed_and_canonical_transfers_agree(dw, Ls):
    """The 4-d K-cycle on the packed and on the canonical layout, both to 1e-10."""
    xs = []
    for layout in (0, 1):
        h, rng, V, dof = _setup(dw, (4, 4, 4, 4), (2, 2, 2, 2), 4, Ls, 2, {"fine_layout": layout, "coarse_tol": 0.4})
        b = _dev(synth.gaussian_complex(rng, (Ls * V * dof,)))
        x = torch.empty_like(b)
        dw.mg_solve(h, b, x, tol=1e-10)
        xs.append(x)
        h.close()
    # |x_0 - x_1| <= 2 * 1e-10 |b| / sigma_min, sigma_min of D_DW above 1e-3 at m = 0.05
    assert float((xs[0] - xs[1]).norm()) <= 2e-7 * float(b.norm())
