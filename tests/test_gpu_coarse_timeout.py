"""A coarse stencil's wait that gave up is reported by the next call on the handle that synchronises,
and by that one only.  The wait is one for a copy that nothing starts, with a limit of 20 ms: no
fault, and the context stays usable."""
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


@pytest.mark.parametrize("solver", [1, 0])
def test_expired_wait_is_reported_once(dw, solver):
    dims, Ls = (8, 8), 4
    rng = synth.rng_for(157)
    U = synth.u1_links(synth.u1_angles(rng, dims, 0.4))
    h = dw.mg_setup(dw.make_geom(dims, Ls), _dev(U), 1.0, 0.1, {"coarse_solver": solver, "coarse_persistent": 0},
                    _dev(synth.gaussian_complex(rng, (8, 128))))
    b = _dev(synth.gaussian_complex(rng, (Ls * 128,)))
    x = torch.empty_like(b)
    rc = _dev(synth.gaussian_complex(rng, (h.coarse_size,)), torch.complex64)
    ec = torch.empty_like(rc)
    v = b.to(torch.complex64)
    calls = [lambda: dw.mg_solve(h, b, x), lambda: dw.mg_coarse_solve(h, rc, ec), lambda: dw.mg_transfer_oblique(h, v)]
    if solver == 1:
        calls.append(lambda: dw.mg_solve_batched(h, torch.cat([b, b]), torch.cat([x, x]), 2))
    for call in calls:
        dw.mg_check_wait_timeout(h, 0.02)
        with pytest.raises(dw.DwfError) as e:
            call()
        assert e.value.status == 4                       # DWF_ERR_TIMEOUT
        assert "timed out" in str(e.value)
        call()                                           # and the handle works on
    h.close()
