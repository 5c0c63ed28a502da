"""What this library is measured on: its public entry points at the sizes its workloads use.

The listed cases are the parts a lattice program spends its time in: operator applications
(2-d U(1) and 4-d SU(3), one field and batches, FP64 and FP32 with 16-bit links), the link force
of a gradient, the coarse operator and the wall transfers, and three whole calls: the
differentiable solve (forward and backward), a batch of solves on lattices of different sizes,
and a 4-d solve.  Solves run to 1e-12, the default of the differentiable solve.

`exact` is written in plain torch FP64 from the operator's definition (include/dwf.h).
"""
import math

import numpy as np
import torch

import paper_2004_07732_gb300 as dw

DEV = "cuda"
# Wilson masses of the near-null relaxation for each width of the link distribution
SETUP_MASS = {0.7: -0.3, 0.5: -0.19, 0.214: -0.035}
SETUP_MASS_SU3 = -0.42
SU3_EPS = 0.3
TOL = 1e-12


def listed():
    return [
        # the smallest lattice of the test problems: one application is all latency
        {"name": "apply_u1_32x32x8_f64", "kind": "apply", "group": "u1", "L0": 32, "L1": 32, "Ls": 8, "prec": "f64",
         "op": "dwf", "dagger": False, "anti": False, "M5": 1.0, "mf": 0.01},
        # the lattice that does not fit the cache, in the solver's inner precision
        {"name": "apply_u1_1024x1024x16_l16", "kind": "apply", "group": "u1", "L0": 1024, "L1": 1024, "Ls": 16,
         "prec": "f32_l16", "op": "dwf", "dagger": False, "anti": False, "M5": 1.0, "mf": 0.005},
        # the preconditioned operator in FP64 on a lattice with no round extent, antiperiodic in time
        {"name": "pvdag_u1_250x333x13_f64", "kind": "apply", "group": "u1", "L0": 250, "L1": 333, "Ls": 13,
         "prec": "f64", "op": "pvdag", "dagger": False, "anti": True, "M5": 1.0, "mf": 0.005},
        # 64 sources on three lattice sizes in one launch
        {"name": "batched_u1_64src_l16", "kind": "batched", "nsrc": 64, "La": 64, "Lb": 128, "Lc": 256, "Ls": 16,
         "prec": "f32_l16", "dagger": False, "M5": 1.0, "mf": 0.005},
        # the 4-d operator (adjoint) on fields in the interchange layout
        {"name": "apply_su3_16x16x16x32x16_l16", "kind": "apply", "group": "su3", "L0": 16, "L1": 16, "L2": 16,
         "L3": 32, "Ls": 16, "prec": "f32_l16", "op": "dwf", "dagger": True, "anti": False, "M5": 1.8, "mf": 0.01},
        # the 4-d operator on fields a program keeps in the packed layout
        {"name": "packed_su3_16x16x16x32x16_l16", "kind": "packed", "group": "su3", "L0": 16, "L1": 16, "L2": 16,
         "L3": 32, "Ls": 16, "prec": "f32_l16", "dagger": False, "anti": False, "M5": 1.8, "mf": 0.01},
        # the SU(3) force of a pair of solutions: the backward pass after its adjoint solve
        {"name": "force_su3_12x12x12x24x12_f64", "kind": "force", "group": "su3", "L0": 12, "L1": 12, "L2": 12,
         "L3": 24, "Ls": 12, "anti": True},
        # one vector between the levels and through the coarse operators of a 256^2 hierarchy
        {"name": "coarse_u1_256x256_1vec", "kind": "coarse", "L0": 256, "L1": 256, "Ls": 16, "nrhs": 1,
         "sigma": 0.7, "M5": 1.0, "mf": 0.005},
        # the coarse operator on 64 vectors at once
        {"name": "coarse_u1_256x256_64vec", "kind": "coarse", "L0": 256, "L1": 256, "Ls": 16, "nrhs": 64,
         "sigma": 0.7, "M5": 1.0, "mf": 0.005},
        # a gradient step: d|x|^2 / d theta of x = D^-1 b, both solves by multigrid
        {"name": "grad_u1_256x256x16", "kind": "grad", "L0": 256, "L1": 256, "Ls": 16, "sigma": 0.7, "M5": 1.0,
         "mf": 0.005},
        # many sources on lattices of three sizes, each size a batch of its own
        {"name": "groups_u1_14src", "kind": "groups", "na": 5, "nb": 5, "nc": 4, "La": 64, "Lb": 128, "Lc": 256,
         "Ls": 16, "sigma": 0.7, "M5": 1.0, "mf": 0.005},
        # a 4-d solve
        {"name": "solve_su3_12x12x12x24x16", "kind": "solve", "group": "su3", "L0": 12, "L1": 12, "L2": 12, "L3": 24,
         "Ls": 16, "M5": 1.8, "mf": 0.01},
    ]


def _log(rng, lo, hi):
    return int(round(math.exp(rng.uniform(math.log(lo), math.log(hi)))))


def draw(rng):
    kind = rng.choice(["apply", "apply", "apply", "apply4", "packed", "batched", "force", "coarse", "coarse", "grad",
                       "groups", "solve"])
    precs = ["f64", "f32", "f32_l16", "f32_lbf16"]
    if kind == "apply":
        return {"kind": "apply", "group": "u1", "L0": _log(rng, 8, 1024), "L1": _log(rng, 8, 1024),
                "Ls": rng.randint(4, 16), "prec": rng.choice(precs), "op": rng.choice(["dwf", "dwf", "pv", "pvdag"]),
                "dagger": rng.random() < 0.5, "anti": rng.random() < 0.5, "M5": 1.0,
                "mf": rng.choice([0.005, 0.01, 0.05])}
    if kind in ("apply4", "packed"):
        odd = 1 if kind == "apply4" else 2
        return {"kind": "apply" if kind == "apply4" else "packed", "group": "su3", "L0": rng.randint(4, 16),
                "L1": rng.randint(4, 16), "L2": rng.randint(4, 16), "L3": _log(rng, 4, 32),
                "Ls": odd * rng.randint(4 // odd, 16 // odd),
                "prec": rng.choice(precs if kind == "apply4" else precs[1:]), "dagger": rng.random() < 0.5,
                "anti": rng.random() < 0.5, "M5": 1.8, "mf": 0.01, **({"op": "dwf"} if kind == "apply4" else {})}
    if kind == "batched":
        return {"kind": "batched", "nsrc": _log(rng, 1, 64), "La": _log(rng, 16, 64), "Lb": _log(rng, 32, 128),
                "Lc": _log(rng, 64, 256), "Ls": rng.randint(4, 16), "prec": rng.choice(precs[1:]),
                "dagger": rng.random() < 0.5, "M5": 1.0, "mf": rng.choice([0.005, 0.01])}
    if kind == "force":
        if rng.random() < 0.5:
            return {"kind": "force", "group": "u1", "L0": _log(rng, 16, 256), "L1": _log(rng, 16, 256),
                    "Ls": rng.randint(4, 16), "anti": rng.random() < 0.5}
        return {"kind": "force", "group": "su3", "L0": rng.randint(4, 12), "L1": rng.randint(4, 12),
                "L2": rng.randint(4, 12), "L3": rng.randint(4, 24), "Ls": rng.randint(4, 12),
                "anti": rng.random() < 0.5}
    if kind == "coarse":
        return {"kind": "coarse", "L0": 4 * rng.randint(4, 64), "L1": 4 * rng.randint(4, 64), "Ls": rng.randint(4, 16),
                "nrhs": rng.choice([1, _log(rng, 2, 64)]), "sigma": rng.choice([0.7, 0.5, 0.214]), "M5": 1.0,
                "mf": rng.choice([0.005, 0.01])}
    if kind == "grad":
        return {"kind": "grad", "L0": 4 * _log(rng, 8, 48), "L1": 4 * _log(rng, 8, 48), "Ls": 2 * rng.randint(4, 8),
                "sigma": rng.choice([0.7, 0.5]), "M5": 1.0, "mf": rng.choice([0.005, 0.01])}
    if kind == "groups":
        return {"kind": "groups", "na": rng.randint(1, 8), "nb": rng.randint(1, 6), "nc": rng.randint(1, 3),
                "La": 4 * rng.randint(8, 16), "Lb": 4 * rng.randint(16, 32), "Lc": 4 * rng.randint(32, 48),
                "Ls": 2 * rng.randint(4, 8), "sigma": rng.choice([0.7, 0.5]), "M5": 1.0, "mf": rng.choice([0.005, 0.01])}
    # (the coarse walls stand for the fine ones only where Ls and the coarse Ls, 4, have one parity)
    return {"kind": "solve", "group": "su3", "L0": 2 * rng.randint(3, 6), "L1": 2 * rng.randint(3, 6),
            "L2": 2 * rng.randint(3, 6), "L3": 2 * rng.randint(4, 10), "Ls": rng.choice([8, 10, 12, 16]), "M5": 1.8,
            "mf": rng.choice([0.01, 0.05])}


# ---------------------------------------------------------------------------
# inputs
# ---------------------------------------------------------------------------
def _dims(c):
    return tuple(c["L%d" % i] for i in range(4 if c.get("group", "u1") == "su3" else 2))


def _gen(seed):
    return torch.Generator(device=DEV).manual_seed(seed)


def _gauss(g, n):
    """n complex numbers, real and imaginary parts N(0, 1)."""
    return torch.view_as_complex(torch.randn(n, 2, dtype=torch.float64, device=DEV, generator=g))


def _su3(g, n):
    """n links exp(i eps H), H the traceless Hermitian part of a complex Gaussian 3 x 3 matrix."""
    a = _gauss(g, 9 * n).view(n, 3, 3)
    h = 0.5 * (a + a.mH)
    h = h - (h.diagonal(dim1=-2, dim2=-1).sum(-1).real / 3)[:, None, None] * torch.eye(3, dtype=a.dtype, device=DEV)
    # a power series of a small multiple, squared back up: every step is a batched product
    x, one = (1j * SU3_EPS / 64) * h, torch.eye(3, dtype=a.dtype, device=DEV).expand(n, 3, 3)
    u = one
    for k in range(12, 0, -1):
        u = one + (x @ u) / k
    for _ in range(6):
        u = u @ u
    return u.reshape(-1)


def _volume(dims):
    return math.prod(dims)


def _anti(c, dims):
    return [0] * (len(dims) - 1) + [1] if c.get("anti") else None


def _geom(c, dims=None):
    dims = dims or _dims(c)
    return dw.make_geom(dims, c.get("Ls", 1), c.get("group", "u1"), _anti(c, dims))


def _fields(c, seed, dims=None, sigma=0.7, n=1):
    """(angles or None, links, n fields) drawn from the seed, complex128."""
    dims = dims or _dims(c)
    g, v = _gen(seed), _volume(dims)
    if len(dims) == 2:
        theta = sigma * torch.randn(2 * v, dtype=torch.float64, device=DEV, generator=g)
        u, dof = torch.polar(torch.ones_like(theta), theta), 2
    else:
        theta, u, dof = None, _su3(g, 4 * v), 12
    return theta, u, [_gauss(g, c["Ls"] * v * dof) for _ in range(n)]


def _classes(c, seed):
    """The lattices of a batch: (dims, sources, seed)."""
    if c["kind"] == "groups":
        counts = [c["na"], c["nb"], c["nc"]]
    else:
        counts = [len(range(k, c["nsrc"], 3)) for k in range(3)]
    return [((L, L), n, 3 * seed + k) for k, (L, n) in enumerate(zip((c["La"], c["Lb"], c["Lc"]), counts)) if n]


def _near_null(c, u, g, steps=30):
    """Eight smooth vectors, as a program keeps them from an earlier gauge field: a few steps of
    CG on D_W D_W^dag v = 0 from Gaussian starts, at the setup mass.  [8][site][spin]"""
    dims, v = _dims(c), _volume(_dims(c))
    op = _Operator(dims, u, -SETUP_MASS[c["sigma"]])
    x = op.inner(_gauss(g, 8 * v * 2), 8)
    r = -op.kernel(op.kernel(x, True), False)
    p, rr = r.clone(), op.norm2(r)
    for _ in range(steps):
        q = op.kernel(op.kernel(p, True), False)
        a = rr / (p.conj() * q).real.flatten(0, -2).sum(0)
        x = x + a * p
        r = r - a * q
        new = op.norm2(r)
        p = r + (new / rr) * p
        rr = new
    return op.canonical(x)


MG_SU3 = {"nvec": 24, "block": [2, 2, 2, 2], "setup_mass": SETUP_MASS_SU3, "post_smooth": 16, "coarse_tol": 0.4}


def prepare(case, seed):
    c, kind = case, case["kind"]
    s = {"case": c}
    if kind in ("apply", "packed"):
        _, u, (psi,) = _fields(c, seed)
        geom, prec = _geom(c), c["prec"]
        psi = psi if prec == "f64" else psi.to(torch.complex64)
        if kind == "packed":
            s.update(U=dw.pack_links(geom, u, prec), psi=dw.pack_spinor(geom, psi))
            s["out"] = torch.zeros_like(s["psi"])
        else:
            s.update(U=dw.links_to(geom, u, prec), psi=psi, out=torch.empty_like(psi))
            if c["op"] == "pvdag":
                s["tmp"] = torch.empty_like(psi)
        s["geom"] = geom
    elif kind == "batched":
        geoms, us, psis = [], [], []
        for dims, n, sd in _classes(c, seed):
            _, u, ps = _fields(c, sd, dims, n=n)
            geom = _geom(c, dims)
            links = dw.links_to(geom, u, c["prec"])
            geoms += [geom] * n
            us += [links] * n
            psis += [p.to(torch.complex64) for p in ps]
        s["outs"] = [torch.empty_like(p) for p in psis]
        s["call"] = dw.BatchedApply(geoms, us, psis, s["outs"], c["prec"])
    elif kind == "force":
        _, u, (lam, x) = _fields(c, seed, n=2)
        s.update(geom=_geom(c), U=u, lam=lam, x=x)
    elif kind == "coarse":
        _, u, _ = _fields(c, seed, sigma=c["sigma"], n=0)
        g = _gen(seed + 1)
        starts = _near_null(c, u, g)
        mg = dw.mg_setup(_geom(c), u, c["M5"], c["mf"], {"setup_mass": SETUP_MASS[c["sigma"]], "setup_maxiter": 0},
                         starts)
        nc = c["nrhs"] * mg.coarse_size
        s.update(mg=mg, v=_gauss(g, nc).to(torch.complex64), out=torch.empty(nc, dtype=torch.complex64, device=DEV))
        if c["nrhs"] == 1:
            s.update(r=_gauss(g, dw.spinor_size(mg.geom)).to(torch.complex64), rc=torch.empty_like(s["v"]),
                     out2=torch.empty_like(s["v"]))
            s["e"] = torch.empty_like(s["r"])
    elif kind == "grad":
        theta, _, (b,) = _fields(c, seed, sigma=c["sigma"])
        geom = _geom(c)
        mg = _hierarchy(c, geom, dw.links_from_angles(geom, theta), seed + 1)
        s.update(geom=geom, mg=mg, theta=theta.requires_grad_(), b=b.requires_grad_())
    elif kind == "groups":
        s.update(mgs=[], bs=[], xs=[], ns=[])
        for dims, n, sd in _classes(c, seed):
            _, u, bs = _fields(c, sd, dims, c["sigma"], n)
            s["mgs"].append(_hierarchy(c, _geom(c, dims), u, sd + 1000003))
            s["bs"].append(torch.cat(bs))
            s["xs"].append(torch.empty_like(s["bs"][-1]))
            s["ns"].append(n)
    else:
        _, u, (b,) = _fields(c, seed)
        g = _gen(seed + 1)
        s["mg"] = dw.mg_setup(_geom(c), u, c["M5"], c["mf"], MG_SU3, _gauss(g, 24 * _volume(_dims(c)) * 12))
        s.update(b=b, x=torch.empty_like(b))
    return s


def _hierarchy(c, geom, u, seed):
    v = geom.L[0] * geom.L[1]
    return dw.mg_setup(geom, u, c["M5"], c["mf"], {"setup_mass": SETUP_MASS[c["sigma"]]}, _gauss(_gen(seed), 8 * v * 2))


def run(state):
    s, c = state, state["case"]
    kind = c["kind"]
    if kind == "apply":
        if c["op"] == "pvdag":
            return dw.dwf_pvdag_apply(s["geom"], s["U"], s["psi"], s["tmp"], s["out"], c["M5"], c["mf"], c["prec"])
        if c["op"] == "pv":
            return dw.pv_apply(s["geom"], s["U"], s["psi"], s["out"], c["M5"], c["dagger"], c["prec"])
        return dw.dwf_apply(s["geom"], s["U"], s["psi"], s["out"], c["M5"], c["mf"], c["dagger"], c["prec"])
    if kind == "packed":
        return dw.dwf_apply_packed(s["geom"], s["U"], s["psi"], s["out"], c["M5"], c["mf"], c["dagger"], c["prec"])
    if kind == "batched":
        return s["call"](c["M5"], c["mf"], c["dagger"])
    if kind == "force":
        return dw.link_force(s["geom"], s["U"], s["lam"], s["x"])
    if kind == "coarse":
        if c["nrhs"] > 1:
            return dw.mg_coarse_apply_multi(s["mg"], s["v"], s["out"], c["nrhs"], c["mf"])
        # down, D_DW and D_PV^dag on the coarse level, and up
        return {"restricted": dw.mg_restrict(s["mg"], s["r"], s["rc"]),
                "dwf": dw.mg_coarse_apply(s["mg"], s["v"], s["out"], c["mf"]),
                "pvdag": dw.mg_coarse_apply(s["mg"], s["v"], s["out2"], 1.0, True),
                "prolonged": dw.mg_prolong(s["mg"], s["v"], s["e"])}
    if kind == "grad":
        x = dw.solve(s["theta"], s["b"], s["geom"], c["M5"], c["mf"], tol=TOL, mg=s["mg"])
        gt, gb = torch.autograd.grad((x.abs() ** 2).sum(), (s["theta"], s["b"]))
        return {"x": x.detach(), "grad_theta": gt, "grad_b": gb}
    if kind == "groups":
        dw.mg_solve_groups(s["mgs"], s["bs"], s["xs"], s["ns"], tol=TOL)
        return s["xs"]
    dw.mg_solve(s["mg"], s["b"], s["x"], tol=TOL)
    return s["x"]


# ---------------------------------------------------------------------------
# work
# ---------------------------------------------------------------------------
def work(case):
    """Fields and links read once, results written once; flops of one application of the operator
    (each U(1) site and slice about 60, each SU(3) one 1320 + 48), of a solve too, whose step
    count the path does not fix."""
    c, kind = case, case["kind"]

    def op(dims, prec="f64", n=1):
        v, dof = _volume(dims), 2 if len(dims) == 2 else 12
        spinor = v * c["Ls"] * dof * (16 if prec == "f64" else 8)
        links = v * len(dims) * (1 if dof == 2 else 9) * {"f64": 16, "f32": 8}.get(prec, 4)
        return n * 2 * spinor + links, n * v * c["Ls"] * (60 if dof == 2 else 1368)

    if kind in ("apply", "packed"):
        b, f = op(_dims(c), c["prec"])
        return {"bytes": b, "flops": f * (2 if c.get("op") == "pvdag" else 1)}
    if kind in ("batched", "groups"):
        both = [op(dims, c.get("prec", "f64"), n) for dims, n, _ in _classes(c, 0)]
        return {"bytes": sum(b for b, _ in both), "flops": sum(f for _, f in both)}
    if kind == "force":
        b, f = op(_dims(c))
        v, nd = _volume(_dims(c)), len(_dims(c))
        return {"bytes": b + (4 * 9 * 16 * v if nd == 4 else 2 * 8 * v),
                "flops": v * nd * c["Ls"] * (24 if nd == 2 else 2 * (24 + 2 * 9 * 8))}
    if kind == "coarse":
        vc, cols = c["L0"] * c["L1"] // 16, 4 * c["nrhs"]
        applies = 2 if c["nrhs"] == 1 else 1
        # FP16 blocks, complex64 vectors
        b, f = vc * (5 * 256 * 4 + (1 + applies) * cols * 16 * 8), applies * vc * cols * 5 * 256 * 8
        if c["nrhs"] == 1:
            # the walls read and the whole vectors written, and the FP32 prolongator
            v = c["L0"] * c["L1"]
            b += v * 2 * 8 * 8 + v * 2 * 8 + vc * cols * 16 * 8 + v * c["Ls"] * 2 * 8
            f += 2 * v * 2 * 8 * 8
        return {"bytes": b, "flops": f}
    b, f = op(_dims(c))
    if kind == "grad":
        b += 2 * op(_dims(c))[0] // 4 + 2 * 8 * 2 * _volume(_dims(c))
        f *= 2
    return {"bytes": b, "flops": f}


# ---------------------------------------------------------------------------
# the same in 64 bits, from the definition
# ---------------------------------------------------------------------------
# gamma_mu as (spin that feeds each spin, factor)
_GAMMA = {2: [([1, 0], [1, 1]), ([1, 0], [-1j, 1j])],
          4: [([3, 2, 1, 0], [-1j, -1j, 1j, 1j]), ([3, 2, 1, 0], [-1, 1, 1, -1]),
              ([2, 3, 0, 1], [-1j, 1j, 1j, -1j]), ([2, 3, 0, 1], [1, 1, 1, 1])]}


class _Operator:
    """D_W(-M5) and D_DW on fields [x_{nd-1}]...[x_0][color][spin][s][column]."""

    def __init__(self, dims, u, M5, Ls=1, mf=0.0, anti=None):
        self.dims, self.nd, self.Ls, self.mf, self.M5 = dims, len(dims), Ls, mf, M5
        self.nc, self.ns = (1, 2) if self.nd == 2 else (3, 4)
        self.u = u.to(torch.complex128).view(self.nd, *reversed(dims), self.nc, self.nc).clone()
        for mu in range(self.nd):
            if anti and anti[mu]:
                self.u[mu].select(self.axis(mu), dims[mu] - 1).mul_(-1)
        self.gamma = [(torch.tensor(p, device=DEV), torch.tensor(f, dtype=torch.complex128, device=DEV)[:, None, None])
                      for p, f in _GAMMA[self.nd]]
        self.back = [torch.roll(self.u[mu], 1, self.axis(mu)).mH.contiguous() for mu in range(self.nd)]
        # the weight of the hop that crosses the walls
        self.up = torch.ones(Ls, 1, dtype=torch.float64, device=DEV)
        self.up[-1] = -mf
        self.down = torch.flip(self.up, (0,))

    def axis(self, mu):
        return self.nd - 1 - mu

    def inner(self, f, columns=1):
        """canonical [column][s][site][spin][color] -> the layout of this class"""
        v = f.to(torch.complex128).view(columns, -1, *reversed(self.dims), self.ns, self.nc)
        k = self.nd
        return v.permute(*range(2, 2 + k), 3 + k, 2 + k, 1, 0).contiguous()

    def canonical(self, f):
        k = self.nd
        return f.permute(k + 3, k + 2, *range(k), k + 1, k).reshape(-1)

    def norm2(self, f):
        return f.abs().square().flatten(0, -2).sum(0)

    def times(self, u, f):
        if self.nc == 1:
            return u[..., None, None] * f
        return (u @ f.flatten(-3)).view_as(f)

    def spin(self, mu, f):
        perm, fac = self.gamma[mu]
        return f.index_select(-3, perm) * fac

    def kernel(self, f, dagger):
        out = (self.nd - self.M5) * f
        sign = -1 if dagger else 1
        for mu in range(self.nd):
            ax = self.axis(mu)
            a = self.times(self.u[mu], torch.roll(f, -1, ax))
            b = self.times(self.back[mu], torch.roll(f, 1, ax))
            out.add_(a + b, alpha=-0.5).add_(self.spin(mu, a - b), alpha=0.5 * sign)
        return out

    def apply(self, f, dagger=False, mf=None):
        up, down = self.up, self.down
        if mf is not None:
            up = up.clone()
            up[-1] = -mf
            down = torch.flip(up, (0,))
        out = self.kernel(f, dagger) + f
        h = self.ns // 2
        above, below = torch.roll(f, -1, -2) * up, torch.roll(f, 1, -2) * down
        plus, minus = (above, below) if dagger else (below, above)
        out[..., :h, :, :] += plus[..., :h, :, :]
        out[..., h:, :, :] += minus[..., h:, :, :]
        return out

    def solve(self, b, dagger=False, tol=2e-15, most=20000):
        """D x = b (or D^dag x = b) by CG on the normal equations, every column with its own
        scalars; restarted from the true residual until that is at its floor."""
        x, r = torch.zeros_like(b), b.clone()
        bn = self.norm2(b)
        last = math.inf
        for _ in range(6):
            z = self.apply(r, not dagger)
            p, rr = z.clone(), self.norm2(z)
            e = torch.zeros_like(b)

            def step():
                q = self.apply(p, dagger)
                a = rr / self.norm2(q)
                e.add_(a * p)
                r.sub_(a * q)
                z = self.apply(r, not dagger)
                new = self.norm2(z)
                p.copy_(z + (new / rr) * p)
                rr.copy_(new)

            side = torch.cuda.Stream()
            side.wait_stream(torch.cuda.current_stream())
            with torch.cuda.stream(side):
                step()
            torch.cuda.current_stream().wait_stream(side)
            graph = torch.cuda.CUDAGraph()
            with torch.cuda.graph(graph):
                for _ in range(10):
                    step()
            for k in range(most // 10):
                graph.replay()
                if k % 5 == 4 and float((self.norm2(r) / bn).max()) < max(tol, last * 1e-8) ** 2:
                    break
            del graph
            x += e
            r = b - self.apply(x, dagger)
            now = float((self.norm2(r) / bn).max()) ** 0.5
            if now < 1e-14 or now > 0.3 * last:
                break
            last = now
        return x

    def link_gradient(self, lam, x):
        """-1/2 sum_s [lam(y) ((1 - gamma) x(y + mu))^dag + ((1 + gamma) x(y)) lam(y + mu)^dag], [mu][site][a][b]"""
        out = []
        for mu in range(self.nd):
            ax = self.axis(mu)
            xf, lf = torch.roll(x, -1, ax), torch.roll(lam, -1, ax)
            a = lam.flatten(-3) @ (xf - self.spin(mu, xf)).flatten(-3).mH
            a += (x + self.spin(mu, x)).flatten(-3) @ lf.flatten(-3).mH
            out.append(-0.5 * a)
        return torch.stack(out)


def _force(op, u, lam, x, anti):
    g = op.link_gradient(lam, x)
    if anti:
        g[-1].select(0, op.dims[-1] - 1).mul_(-1)
    u = u.view_as(g)
    if op.nc == 1:
        return (g.conj() * 1j * u).real.reshape(-1)
    f = 1j * u @ g.mH
    f = 0.5 * (f + f.mH)
    tr = f.diagonal(dim1=-2, dim2=-1).sum(-1) / 3
    return (f - tr[..., None, None] * torch.eye(3, dtype=f.dtype, device=DEV)).reshape(-1)


def _rounded(u, prec):
    """Links as their storage holds them.  numpy rounds FP64 to FP16 once; torch goes by FP32."""
    if prec == "f64":
        return u
    if prec == "f32_l16":
        half = torch.view_as_real(u).cpu().numpy().astype(np.float16)
        return torch.view_as_complex(torch.from_numpy(half.astype(np.float64)).to(DEV))
    to = torch.float32 if prec == "f32" else torch.bfloat16
    return torch.view_as_complex(torch.view_as_real(u).to(to).to(torch.float64))


def _exact_coarse(c, seed):
    dims, sh = _dims(c), (c["L1"], c["L0"])
    _, u, _ = _fields(c, seed, sigma=c["sigma"], n=0)
    g = _gen(seed + 1)
    null = _near_null(c, u, g)
    by, bx = sh[0] // 4, sh[1] // 4
    vc = by * bx

    def blocks(t):       # [..., y, x, ...] with y, x first -> [coarse site][site of it]
        return t.view(by, 4, bx, 4, *t.shape[2:]).transpose(1, 2).reshape(vc, 16, *t.shape[2:])

    # Gram-Schmidt of each aggregate's vectors of each chirality, in vector order, twice over
    q = blocks(null.view(8, *sh, 2).permute(1, 2, 3, 0).contiguous())        # [site][16][chirality][vec]
    for _ in range(2):
        cols = []
        for k in range(8):
            w = q[..., k]
            for o in cols:
                w = w - (o.conj() * w).sum(1, keepdim=True) * o
            cols.append(w / w.abs().square().sum(1, keepdim=True).sqrt())
        q = torch.stack(cols, -1)
    # the prolongator as the library's vectors see it: P psi of coarse [site][chirality][vec]
    n, cols, ls = c["nrhs"], 4 * c["nrhs"], c["Ls"]
    v = _gauss(g, n * 4 * vc * 16).to(torch.complex64).to(torch.complex128).view(n, 4, vc, 2, 8)

    def lift(e):          # [col][coarse site][chirality][vec] -> [col][y][x][chirality]
        f = torch.einsum("sick,nsck->nsic", q, e)
        return f.view(-1, by, bx, 4, 4, 2).transpose(2, 3).reshape(-1, *sh, 2)

    def lower(f):
        f = f.view(-1, by, 4, bx, 4, 2).transpose(2, 3).reshape(-1, vc, 16, 2)
        return torch.einsum("sick,nsic->nsck", q.conj(), f)

    # the Galerkin blocks, column by column: P^dag D_W P on unit vectors; the hops that leave an
    # aggregate go to the neighbours' blocks.  Stored in FP16.
    op = _Operator(dims, u, c["M5"])
    ys = torch.arange(sh[0], device=DEV)[:, None] % 4
    xs = torch.arange(sh[1], device=DEV)[None, :] % 4
    inside = [(xs < 3).to(torch.float64).expand(sh), (ys < 3).to(torch.float64).expand(sh)]
    y = torch.zeros(5, vc, 16, 16, dtype=torch.complex128, device=DEV)
    for col in range(16):
        unit = torch.zeros(1, vc, 2, 8, dtype=torch.complex128, device=DEV)
        unit[0, :, col // 8, col % 8] = 1
        f = op.inner(lift(unit).reshape(-1), 1)
        parts = [torch.zeros_like(f) for _ in range(5)]
        parts[0] += (2 - c["M5"]) * f
        for mu in range(2):
            ax = op.axis(mu)
            a = op.times(op.u[mu], torch.roll(f, -1, ax))
            b = op.times(op.back[mu], torch.roll(f, 1, ax))
            a, b = -0.5 * (a - op.spin(mu, a)), -0.5 * (b + op.spin(mu, b))
            keep = inside[mu][..., None, None, None, None]
            low = torch.roll(keep, 1, ax)
            parts[0] += keep * a + low * b
            parts[1 + 2 * mu] += (1 - keep) * a
            parts[2 + 2 * mu] += (1 - low) * b
        for d in range(5):
            y[d, :, :, col] = lower(op.canonical(parts[d]).view(1, *sh, 2)).view(vc, 16)
    y = _rounded(y, "f32_l16")
    sigma = torch.tensor([1.0] * 8 + [-1.0] * 8, dtype=torch.float64, device=DEV)

    def coarse(w, mf, dagger):
        z = w.reshape(n, 4, by, bx, 16)
        s3 = sigma if dagger else torch.ones_like(sigma)
        k = z * s3
        hops = [k, torch.roll(k, -1, 3), torch.roll(k, 1, 3), torch.roll(k, -1, 2), torch.roll(k, 1, 2)]
        out = sum(torch.einsum("sab,nlsb->nlsa", y[d], hops[d].reshape(n, 4, vc, 16)) for d in range(5)) * s3
        z = w.reshape(n, 4, vc, 16)
        up = torch.ones(4, 1, 1, dtype=torch.float64, device=DEV)
        up[3] = -mf
        above, below = torch.roll(z, -1, 1) * up, torch.roll(z, 1, 1) * torch.flip(up, (0,))
        plus, minus = (above, below) if dagger else (below, above)
        out = out + z
        out[..., :8] += plus[..., :8]
        out[..., 8:] += minus[..., 8:]
        return out.reshape(-1)

    if n > 1:
        return coarse(v, c["mf"], False)
    r = _gauss(g, ls * _volume(dims) * 2).to(torch.complex64).to(torch.complex128).view(ls, *sh, 2)
    walls = torch.stack([r[ls - 1, ..., 0], r[0, ..., 1]], -1)
    low = lower(walls[None])[0]
    rc = torch.zeros(4, vc, 2, 8, dtype=torch.complex128, device=DEV)
    rc[3, :, 0], rc[0, :, 1] = low[:, 0], low[:, 1]
    e = lift(torch.stack([v[0, 3, :, 0], v[0, 0, :, 1]], 1)[None])[0]
    up = torch.zeros(ls, *sh, 2, dtype=torch.complex128, device=DEV)
    up[ls - 1, ..., 0], up[0, ..., 1] = e[..., 0], e[..., 1]
    return {"restricted": rc.reshape(-1), "dwf": coarse(v, c["mf"], False), "pvdag": coarse(v, 1.0, True),
            "prolonged": up.reshape(-1)}


def exact(case, seed):
    c, kind = case, case["kind"]
    if kind in ("apply", "packed"):
        dims = _dims(c)
        _, u, (psi,) = _fields(c, seed)
        psi = psi if c["prec"] == "f64" else psi.to(torch.complex64)
        op = _Operator(dims, _rounded(u, c["prec"]), c["M5"], c["Ls"], c["mf"], _anti(c, dims))
        f, what = op.inner(psi), c.get("op", "dwf")
        if what == "pvdag":
            f = op.apply(op.apply(f), True, 1.0)
        else:
            f = op.apply(f, c["dagger"], 1.0 if what == "pv" else None)
        out = op.canonical(f)
        if kind == "packed":
            v, nb = _volume(dims), -(-_volume(dims) // 32)
            p = torch.zeros(c["Ls"], 32 * nb, 12, dtype=out.dtype, device=DEV)
            p[:, :v] = out.view(c["Ls"], v, 12)
            out = p.view(c["Ls"] // 2, 2, nb, 32, 12).permute(0, 2, 4, 3, 1).reshape(-1)
        return out
    if kind == "batched":
        outs = []
        for dims, n, sd in _classes(c, seed):
            _, u, ps = _fields(c, sd, dims, n=n)
            op = _Operator(dims, _rounded(u, c["prec"]), c["M5"], c["Ls"], c["mf"])
            outs += [op.canonical(op.apply(op.inner(p.to(torch.complex64)), c["dagger"])) for p in ps]
        return outs
    if kind == "force":
        _, u, (lam, x) = _fields(c, seed, n=2)
        op = _Operator(_dims(c), u, 1.0, c["Ls"])
        return _force(op, u, op.inner(lam), op.inner(x), c["anti"])
    if kind == "coarse":
        return _exact_coarse(c, seed)
    if kind == "grad":
        theta, u, (b,) = _fields(c, seed, sigma=c["sigma"])
        op = _Operator(_dims(c), u, c["M5"], c["Ls"], c["mf"])
        x = op.solve(op.inner(b))
        lam = op.solve(2 * x, True)
        return {"x": op.canonical(x), "grad_theta": -_force(op, u, lam, x, False), "grad_b": op.canonical(lam)}
    if kind == "groups":
        return None      # well over a minute: every source is a solve of its own
    _, u, (b,) = _fields(c, seed)
    op = _Operator(_dims(c), u, c["M5"], c["Ls"], c["mf"])
    return op.canonical(op.solve(op.inner(b)))
