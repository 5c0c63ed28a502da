"""Rounding errors of the fine operators against an evaluation in the operator's own precision with
every sum and product of the definition apart (a complex product: two products, one of them
fused into the sum), emulated on the host: the kernels fuse and reorder, and may not be further
from the exact result for it.  Errors are root mean squares over the components, relative to
the result; the exact result is the same evaluation in the wider type."""
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


class _Arithmetic:
    """Complex arrays [2 (re, im)]... in the wide type, every operation rounded to the narrow one"""

    def __init__(self, wide, narrow):
        self.wide, self.narrow = wide, narrow

    def r(self, x):
        return x.astype(self.narrow).astype(self.wide) if self.narrow else x

    def add(self, a, b):
        return self.r(a + b)

    def mul(self, a, b, conj=False):
        y = -a[1] if conj else a[1]
        return np.stack([self.r(a[0] * b[0] - self.r(y * b[1])), self.r(a[0] * b[1] + self.r(y * b[0]))])

    def axpy(self, s, a, b):
        return self.r(s * a + b)


def _i(a, n=1):
    """i^n a"""
    return [a, np.stack([-a[1], a[0]]), -a, np.stack([a[1], -a[0]])][n % 4]


# gamma_mu = [[0, A], [A^dag, 0]]: (power of i, column) of every row of A
_A = {2: [[(0, 0)], [(3, 0)]], 4: [[(3, 1), (3, 0)], [(2, 1), (0, 0)], [(3, 0), (1, 1)], [(0, 0), (0, 1)]]}


def _neighbour(dims, mu, step):
    c = np.indices(tuple(reversed(dims))).reshape(len(dims), -1)[::-1].copy()
    c[mu] = (c[mu] + step) % dims[mu]
    return (c * np.cumprod([1] + list(dims))[:-1][:, None]).sum(0)


def _evaluate(op, dims, U, v, M5, mf, dag):
    """U: [2][mu][site][c][c], v: [2][s][site][spin][c]"""
    nd, half = len(dims), v.shape[3] // 2
    hops = np.zeros_like(v)
    for mu in range(nd):
        A = _A[nd][mu]
        back = {c: (-n % 4, r) for r, (n, c) in enumerate(A)}         # rows of A^dag
        for fwd in (True, False):
            nb = _neighbour(dims, mu, 1 if fwd else -1)
            sign = -1 if fwd != dag else 1
            u = U[:, mu] if fwd else np.swapaxes(U[:, mu][:, nb], -1, -2)
            w = v[:, :, nb]
            h = np.stack([op.add(w[:, :, :, a], sign * _i(w[:, :, :, half + c], n)) for a, (n, c) in enumerate(A)], 3)
            t = np.zeros_like(h)
            for b in range(u.shape[-1]):
                t = op.add(t, op.mul(u[:, None, :, None, :, b], h[..., b][..., None], conj=not fwd))
            hops[:, :, :, :half] = op.add(hops[:, :, :, :half], t)
            low = np.stack([sign * _i(t[:, :, :, back[c][1]], back[c][0]) for c in range(half)], 3)
            hops[:, :, :, half:] = op.add(hops[:, :, :, half:], low)
    below = np.concatenate([op.r(-mf * v[:, -1:]), v[:, :-1]], 1)
    above = np.concatenate([v[:, 1:], op.r(-mf * v[:, :1])], 1)
    plus, minus = (above, below) if dag else (below, above)
    out = op.axpy(op.wide(nd - M5 + 1), v, -hops / 2)
    out[:, :, :, :half] = op.add(out[:, :, :, :half], plus[:, :, :, :half])
    out[:, :, :, half:] = op.add(out[:, :, :, half:], minus[:, :, :, half:])
    return out


def _errors(dw, dims, Ls, group, prec, wide, narrow, dag):
    rng = synth.rng_for(151)
    V, nc, ns = int(np.prod(dims)), 3 if group == "su3" else 1, 4 if group == "su3" else 2
    U = synth.su3_links(rng, dims, 0.7) if nc == 3 else synth.u1_links(synth.u1_angles(rng, dims, 0.7))
    U = np.ascontiguousarray(U).reshape(len(dims), V, nc, nc)
    psi = synth.gaussian_complex(rng, (Ls, V, ns, nc))
    M5, mf = 1.75, float(np.float32(0.01))
    g = dw.make_geom(dims, Ls, group)
    Ud = dw.links_to(g, torch.from_numpy(U.reshape(-1)).to("cuda"), prec)
    p = torch.from_numpy(psi.reshape(-1)).to("cuda").to(dw.spinor_dtype(prec))
    got = dw.dwf_apply(g, Ud, p, torch.empty_like(p), M5, mf, dag, prec).cpu().numpy().reshape(psi.shape)

    def parts(a):
        return np.stack([a.real, a.imag]).astype(narrow).astype(wide)

    exact = _evaluate(_Arithmetic(wide, None), dims, parts(U), parts(psi), M5, mf, dag)
    apart = _evaluate(_Arithmetic(wide, narrow), dims, parts(U), parts(psi), M5, mf, dag)
    norm = np.sqrt((exact ** 2).sum())
    return [float(np.sqrt(((x - exact) ** 2).sum()) / norm) for x in (parts(got), apart)]


@pytest.mark.parametrize("dag", [False, True])
def test_su3_fp32(dw, dag):
    """(products of FP32 numbers are exact in FP64, their sums rounded there 29 bits further down)"""
    kernel, apart = _errors(dw, (8, 8, 8, 8), 6, "su3", "f32", np.float64, np.float32, dag)
    assert kernel <= apart, (kernel, apart)


@pytest.mark.skipif(np.finfo(np.longdouble).nmant < 106, reason="needs a type that holds products of FP64 numbers")
@pytest.mark.parametrize("dag", [False, True])
def test_u1_fp64(dw, dag):
    """(147,456 real components: 0.55% is three standard deviations of a root mean square)"""
    kernel, apart = _errors(dw, (64, 48), 12, "u1", "f64", np.longdouble, np.float64, dag)
    assert kernel <= 1.0055 * apart, (kernel, apart)
