"""The reduction of the blocked GCR where a row's thread blocks meet in two stages (more than ten of
them, the last group not full) and its basis goes over several groups of blocks (from 16 directions
on), and where directions are dropped because the Krylov space ends inside a block.  Against the
two-pass form, which takes one step at a time: both minimise over the same spaces, so outer iterations agree
up to rounding (at most 5% or 2 more), and a coarse solve takes at most the rest of its last block, three
steps, more."""
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


def _dev(a):
    return torch.from_numpy(np.ascontiguousarray(a).reshape(-1)).to("cuda")


def _solve(dw, g, U, starts, b, nrhs, M5, mf, params):
    h = dw.mg_setup(g, _dev(U), M5, mf, params, _dev(starts))
    x = torch.empty_like(b)
    stats, _ = dw.mg_solve_batched(h, b, x, nrhs, tol=1e-10)
    h.close()
    n = b.numel() // nrhs
    for r in range(nrhs):
        y, part = torch.empty(n, dtype=b.dtype, device="cuda"), slice(r * n, (r + 1) * n)
        dw.dwf_apply(g, _dev(U), x[part], y, M5, mf)
        assert float((b[part] - y).norm()) <= 1.0001e-10 * float(b[part].norm())
    return stats


def _compare(one, two):
    for a, b in zip(one, two):
        assert a["iterations"] <= b["iterations"] + max(2, 0.05 * b["iterations"]), (a, b)
        assert a["coarse_avg_iters"] <= 1.05 * b["coarse_avg_iters"] + 3, (a, b)


@pytest.mark.parametrize("nrhs", [1, 2])
def test_groups_of_blocks(dw, nrhs):
    """48 blocks of a fine row (the fifth group has eight), 12 of a coarse one; 21 and 24 directions"""
    dims, Ls = (96, 64), 8
    rng = synth.rng_for(167)
    U = synth.u1_links(synth.u1_angles(rng, dims, 0.4))
    V = dims[0] * dims[1]
    starts = synth.gaussian_complex(rng, (8, V * 2))
    b = _dev(synth.gaussian_complex(rng, (nrhs, Ls * V * 2)))
    params = {"setup_mass": -0.12, "setup_maxiter": 60, "post_smooth": 21, "coarse_restart": 24, "coarse_tol": 0.02}
    runs = [_solve(dw, dw.make_geom(dims, Ls), U, starts, b, nrhs, 1.0, 0.01, {**params, "cgs_passes": p}) for p in (1, 2)]
    _compare(*runs)


@pytest.mark.parametrize("dims,group,Ls", [((8, 8), "u1", 2), ((8, 8), "u1", 3), ((4, 4, 4, 4), "su3", 2)])
def test_exhausted_spaces(dw, dims, group, Ls):
    """Unit links and a source that is constant over the lattice: the operator acts on at most 2 Ls
    numbers, fewer than the smoother's steps, so that blocks lose directions, first ones too."""
    nd, V = len(dims), int(np.prod(dims))
    nc, ns = (3, 4) if group == "su3" else (1, 2)
    U = np.broadcast_to(np.eye(nc, dtype=complex), (nd, V, nc, nc))
    rng = synth.rng_for(173)
    nvec = 8 if group == "u1" else 4
    starts = synth.gaussian_complex(rng, (nvec, V * ns * nc))
    b = np.broadcast_to(synth.gaussian_complex(rng, (Ls, 1, ns, nc)), (Ls, V, ns, nc))
    g = dw.make_geom(dims, Ls, group)
    params = {"nvec": nvec, "setup_mass": -0.05, "setup_maxiter": 20, "post_smooth": 8, "Ls_c": 2}
    if group == "su3":
        params["block"] = [2, 2, 2, 2]
    M5 = 1.0 if group == "u1" else 1.8
    runs = [_solve(dw, g, U, starts, _dev(b), 1, M5, 0.1, {**params, "cgs_passes": p}) for p in (1, 2)]
    _compare(*runs)
