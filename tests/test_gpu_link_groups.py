"""GPU parity of the link force and the link gradient where the slices of one link are split
over groups of threads (1, 2, 4 and 8 groups, slices that do not divide evenly) and where a
lattice extent is 1 or 2, at the 1e-12 of the other FP64 parity tests."""
import numpy as np
import pytest
import torch

import synth
from oracle import force

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


@pytest.mark.parametrize("dims,Ls", [((1, 2), 1), ((5, 3), 3), ((17, 9), 5), ((40, 13), 17)])
def test_u1_slice_groups(dw, dims, Ls):
    rng = synth.rng_for(71)
    V, anti = int(np.prod(dims)), [0, 1]
    U = synth.u1_links(synth.u1_angles(rng, dims, 0.6))
    lam, x = (synth.gaussian_spinor(rng, dims, Ls) for _ in range(2))
    g = dw.make_geom(dims, Ls, antiperiodic=anti)
    F = dw.link_force(g, _dev(U), _dev(lam), _dev(x)).cpu().numpy().reshape(2, V)
    G = dw.link_grad(g, _dev(lam), _dev(x)).cpu().numpy().reshape(2, V)
    want = force.link_derivative_contraction(U, dims, Ls, lam, x, anti)
    scale = np.abs(want).max()
    assert np.abs(F - want).max() <= 1e-12 * scale
    # along the angle: dU = i U
    assert np.abs((np.conj(G) * 1j * U).real - want).max() <= 1e-12 * scale


@pytest.mark.parametrize("dims,Ls", [((1, 2, 3, 2), 1), ((3, 2, 2, 5), 2), ((2, 3, 4, 2), 9), ((2, 2, 3, 3), 17)])
def test_su3_slice_groups(dw, dims, Ls):
    rng = synth.rng_for(72)
    V, anti = int(np.prod(dims)), [0, 1, 0, 1]
    U = synth.su3_links(rng, dims, 0.4)
    lam, x = (synth.gaussian_spinor(rng, dims, Ls, "su3") for _ in range(2))
    g = dw.make_geom(dims, Ls, group="su3", antiperiodic=anti)
    F = dw.link_force(g, _dev(U), _dev(lam), _dev(x)).cpu().numpy().reshape(4, V, 3, 3)
    G = dw.link_grad(g, _dev(lam), _dev(x)).cpu().numpy().reshape(4, V, 3, 3)
    links = [(mu, int(s)) for mu in range(4) for s in (0, V // 2, V - 1)]
    want = force.link_force_su3(U, dims, Ls, lam, x, links, anti)
    got = np.array([F[k] for k in links])
    assert np.abs(got - want).max() <= 1e-12 * np.abs(want).max()
    # F is the traceless Hermitian part of i U G^dag
    A = np.array([1j * U[k] @ G[k].conj().T for k in links])
    A = 0.5 * (A + np.conj(np.swapaxes(A, -1, -2)))
    A -= np.trace(A, axis1=-2, axis2=-1)[:, None, None] / 3 * np.eye(3)
    assert np.abs(A - want).max() <= 1e-12 * np.abs(want).max()
