"""Infinite inputs of the 2-d operator: a component that is infinite on one site and slice reaches its
neighbours as the infinities that the sums of the definition give, in FP64 as in FP32.  The four
neighbours see it through one hop each, whose other inputs are finite, so nothing there is NaN."""
import numpy as np
import pytest
import torch

import synth

pytestmark = pytest.mark.gpu
DIMS, LS, S, X, Y = (7, 6), 5, 2, 3, 4


@pytest.fixture(scope="module")
def dw():
    if not torch.cuda.is_available():
        pytest.skip("no GPU")
    import paper_2004_07732_gb300 as pkg
    pkg.lib()
    return pkg


@pytest.mark.parametrize("prec", ["f64", "f32"])
@pytest.mark.parametrize("dag", [False, True])
@pytest.mark.parametrize("spin", [0, 1])
def test_one_infinite_component(dw, prec, dag, spin):
    V = DIMS[0] * DIMS[1]
    rng = synth.rng_for(149)
    theta = rng.uniform(0.2, 1.2, (2, V))                      # no link with a zero part
    U = np.exp(1j * theta)
    psi = synth.gaussian_complex(rng, (LS, V, 2))
    g = dw.make_geom(DIMS, LS)
    site = X + DIMS[0] * Y
    outs = []
    for value in (1.0, 2.0, np.inf):
        v = psi.copy()
        v[S, site, spin] = complex(value, psi[S, site, spin].imag)
        p = torch.from_numpy(v.reshape(-1)).to("cuda").to(dw.spinor_dtype(prec))
        Ud = dw.links_to(g, torch.from_numpy(U.reshape(-1)).to("cuda"), prec)
        outs.append(dw.dwf_apply(g, Ud, p, torch.empty_like(p), 1.0, 0.05, dag, prec).cpu().numpy().reshape(LS, V, 2))
    one, two, inf = outs
    nbs = [(X + 1) % DIMS[0] + DIMS[0] * Y, X - 1 + DIMS[0] * Y, X + DIMS[0] * ((Y + 1) % DIMS[1]), X + DIMS[0] * (Y - 1)]
    for nb in nbs:
        # every real number there moves with the component, and so becomes an infinity of that sign
        got, want = inf[S, nb].view(inf.real.dtype), (two - one)[S, nb].view(inf.real.dtype)
        assert np.all(np.abs(want) > 0.05)
        assert np.array_equal(got, np.where(want > 0, np.inf, -np.inf))
    touched = np.zeros((LS, V), bool)
    touched[S, nbs] = touched[S, site] = True
    touched[[S - 1, S + 1], site] = True
    assert np.array_equal(inf[~touched], one[~touched])
