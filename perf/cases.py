"""The work that users of the solver have it do, as timed cases.

A case is one pass through the public entry points: an operator or transfer
applied to a vector, a whole solve on a handle whose deflation space exists, or
a cold start (set-up and solve of a new configuration).  Gauge fields are
quenched U(1) fields at beta = 6.0 made here from the seed; right-hand sides are
complex Gaussian, as in the benchmark and the tests.
"""
import math

import torch

import paper_1912_02868_gb300 as mg

BETA = 6.0
# The smallest real part of the spectrum of D(0) on beta = 6.0 fields lies
# between 0.058 and 0.087, so this mass leaves a gap of about 1e-2 on every
# field without tuning it per field (the mass-gap study covers 1e-1 to 1e-4).
M0 = -0.05
# Solves whose solution, and not only its residual, is wanted to 1e-10 (the
# tolerance range of the solution-accuracy tests).
TOL = 1e-11
NV = 12

PRECISION = {"fp64": mg.MG_FP64, "mixed": mg.MG_MIXED, "bf16": mg.MG_MIXED_BF16, "fp16": mg.MG_MIXED_FP16}
BLOCK_PRECISION = {"bf16": mg.MG_BF16, "fp16": mg.MG_F16}


def listed():
    return [
        # one fine apply on the smallest lattice of the benchmark: launch latency
        {"name": "wilson 64 f64", "kind": "wilson", "Lx": 64, "Lt": 64, "dtype": "f64", "dagger": False},
        # the fine apply from HBM, the size of the benchmark's fine roofline
        {"name": "wilson 2048 f32", "kind": "wilson", "Lx": 2048, "Lt": 2048, "dtype": "f32", "dagger": False},
        # the intermediate operator of a 512^2 lattice, larger than L2
        {"name": "stencil 512 f32", "kind": "stencil", "Lx": 512, "Lt": 512, "level": 1, "dtype": "f32",
         "dagger": False},
        # both coarsenings, down and up, of a 512^2 lattice
        {"name": "transfer 512 f32", "kind": "transfer", "Lx": 512, "Lt": 512, "dtype": "f32"},
        # the tensor-core block products of a 16-right-hand-side block
        {"name": "block 512 fp16 x16", "kind": "block", "Lx": 512, "Lt": 512, "level": 1, "dtype": "fp16",
         "nrhs": 16},
        # the plain FP64 method on 64^2, one right-hand side
        {"name": "solve 64 fp64", "kind": "solve", "Lx": 64, "Lt": 64, "precision": "fp64", "nrhs": 1,
         "parallel": 1, "partial": 0.0},
        # the headline path: mixed precision on 256^2, one right-hand side
        {"name": "solve 256 mixed", "kind": "solve", "Lx": 256, "Lt": 256, "precision": "mixed", "nrhs": 1,
         "parallel": 1, "partial": 0.0},
        # the same from a lattice whose coarsest grid outgrows one cluster's shared memory
        {"name": "solve 384 mixed", "kind": "solve", "Lx": 384, "Lt": 384, "precision": "mixed", "nrhs": 1,
         "parallel": 1, "partial": 0.0},
        # several right-hand sides on concurrent solve contexts
        {"name": "solve 256 mixed x7 parallel", "kind": "solve", "Lx": 256, "Lt": 256, "precision": "mixed",
         "nrhs": 7, "parallel": 7, "partial": 0.0},
        # the batched solve of 64 right-hand sides
        {"name": "solve 256 bf16 x64", "kind": "solve", "Lx": 256, "Lt": 256, "precision": "bf16", "nrhs": 64,
         "parallel": 1, "partial": 0.0},
        # the partial intermediate solve
        {"name": "solve 128 partial", "kind": "solve", "Lx": 128, "Lt": 128, "precision": "mixed", "nrhs": 1,
         "parallel": 1, "partial": 0.2},
        # a new configuration on a ragged lattice: set-up, deflation build, three right-hand sides
        {"name": "cold 80x48 mixed", "kind": "cold", "Lx": 80, "Lt": 48, "precision": "mixed", "nrhs": 3},
    ]


def _log_int(rng, lo, hi):
    return int(round(math.exp(rng.uniform(math.log(lo), math.log(hi)))))


def _extent(rng, lo, hi):
    """A lattice extent of a hierarchy: a multiple of 16."""
    return 16 * max(1, _log_int(rng, lo / 16, hi / 16))


def draw(rng):
    kind = rng.choice(["wilson", "wilson", "stencil", "transfer", "block", "solve", "solve", "solve", "cold"])
    if kind == "wilson":
        # any extents from 16 up, odd ones among them
        return {"kind": kind, "Lx": _log_int(rng, 16, 2048), "Lt": _log_int(rng, 16, 2048),
                "dtype": rng.choice(["f64", "f32"]), "dagger": rng.random() < 0.5}
    if kind in ("stencil", "transfer", "block"):
        case = {"kind": kind, "Lx": _extent(rng, 32, 512), "Lt": _extent(rng, 32, 512)}
        if kind == "block":
            case.update(level=rng.choice([1, 2]), dtype=rng.choice(["bf16", "fp16"]),
                        nrhs=8 * rng.randint(1, 8 if case["Lx"] * case["Lt"] <= 256 * 256 else 2))
        else:
            case["dtype"] = rng.choice(["f64", "f32"])
        if kind == "stencil":
            case.update(level=rng.choice([1, 2]), dagger=rng.random() < 0.5)
        return case
    if kind == "cold":
        return {"kind": kind, "Lx": _extent(rng, 32, 96), "Lt": _extent(rng, 32, 96),
                "precision": rng.choice(["fp64", "mixed"]), "nrhs": rng.randint(1, 3)}
    precision = rng.choice(["fp64", "mixed", "mixed", "bf16", "fp16"])
    case = {"kind": kind, "Lx": _extent(rng, 32, 256 if precision == "fp64" else 320),
            "Lt": _extent(rng, 32, 256 if precision == "fp64" else 320), "precision": precision, "nrhs": 1,
            "parallel": 1, "partial": 0.0}
    if precision in ("bf16", "fp16"):
        case["nrhs"] = _log_int(rng, 2, 48)
    elif precision == "mixed":
        case["nrhs"] = rng.choice([1, 1, 2, 5])
        case["parallel"] = rng.choice([1, case["nrhs"]])
        case["partial"] = rng.choice([0.0, 0.0, 0.2])
    return case


# ------------------------------------------------------------------ inputs ---


def _generator(seed, tag):
    g = torch.Generator(device="cpu")
    g.manual_seed(1000003 * (int(seed) % (1 << 40)) + tag)
    return g


def _gauss(shape, seed, tag, dtype=torch.complex128):
    """Complex Gaussian, E|z|^2 = 1, on the GPU."""
    g = torch.Generator(device="cuda")
    g.manual_seed(1000003 * (int(seed) % (1 << 40)) + tag)
    return torch.randn(shape, dtype=torch.complex128, device="cuda", generator=g).to(dtype)


def _gauge(Lx, Lt, seed):
    """U(1) field complex128[Lt][Lx][2] of the Wilson plaquette action at BETA.

    In two dimensions the plaquette angles are independent von Mises variables up
    to the constraint on their sum: they are drawn so and shifted to sum to zero,
    links that have them are built row by row, with random holonomies, and a
    random gauge transformation is applied.
    """
    g = _generator(seed, 1)
    n = 1 << 14
    edges = torch.linspace(-math.pi, math.pi, n + 1, dtype=torch.float64)
    cdf = torch.cumsum(torch.exp(BETA * (torch.cos((edges[1:] + edges[:-1]) / 2) - 1)), 0)
    cdf = torch.cat([torch.zeros(1, dtype=torch.float64), cdf / cdf[-1]])
    u = torch.rand(Lt * Lx, generator=g, dtype=torch.float64)
    k = (torch.searchsorted(cdf, u, right=True) - 1).clamp(0, n - 1)
    theta = edges[k] + (u - cdf[k]) / (cdf[k + 1] - cdf[k]) * (edges[1] - edges[0])
    theta = (theta - theta.mean()).reshape(Lt, Lx)
    row = theta.sum(1, keepdim=True) / Lx
    at = torch.cumsum(theta - row, 1)
    at = torch.cat([torch.zeros(Lt, 1, dtype=torch.float64), at[:, :-1]], 1)
    ax = -torch.cat([torch.zeros(1, 1, dtype=torch.float64), torch.cumsum(row, 0)[:-1]], 0).expand(Lt, Lx)
    hol = 2 * math.pi * torch.rand(2, generator=g, dtype=torch.float64)
    w = 2 * math.pi * torch.rand(Lt, Lx, generator=g, dtype=torch.float64)
    ax = ax + hol[0] / Lx + w - torch.roll(w, -1, 1)
    at = at + hol[1] / Lt + w - torch.roll(w, -1, 0)
    ang = torch.stack([ax, at], -1)
    return torch.polar(torch.ones_like(ang), ang).cuda()


def _null_vectors(Lx, Lt, seed):
    """Near-null vectors a program loads with a saved hierarchy, for the operator
    cases (their arithmetic does not depend on how null the vectors are)."""
    return (_gauss((NV, Lt, Lx, 2), seed, 2), _gauss((NV, Lt // 4, Lx // 4, 24), seed, 3))


def _level_shape(case, level):
    f = 4 ** level
    return (case["Lt"] // f, case["Lx"] // f, 2 if level == 0 else 24)


def _cdtype(name):
    return torch.complex128 if name == "f64" else torch.complex64


def _operands(case, seed):
    """The vectors of an operator, transfer or block case."""
    if case["kind"] == "transfer":
        dt = _cdtype(case["dtype"])
        return [_gauss(_level_shape(case, level), seed, 10 + i, dt) for i, level in enumerate((0, 1, 1, 2))]
    if case["kind"] == "block":
        return [_gauss((case["nrhs"],) + _level_shape(case, case["level"]), seed, 10, torch.complex64)]
    return [_gauss(_level_shape(case, case.get("level", 0)), seed, 10, _cdtype(case["dtype"]))]


def _rhs(case, seed):
    return _gauss((case["nrhs"], case["Lt"], case["Lx"], 2), seed, 20)


def prepare(case, seed):
    Lx, Lt, kind = case["Lx"], case["Lt"], case["kind"]
    U = _gauge(Lx, Lt, seed)
    st = {"case": case, "U": U}
    if kind == "wilson":
        st["U"] = U.to(_cdtype(case["dtype"]))
        st["x"] = _operands(case, seed)[0]
        st["y"] = torch.empty_like(st["x"])
        return st
    if kind in ("stencil", "transfer", "block"):
        nv0, nv1 = _null_vectors(Lx, Lt, seed)
        params = mg.default_params(precision=PRECISION["mixed"])
        st["h"] = mg.mg_setup_from_vectors(U, Lx, Lt, M0, nv0, nv1, params=params)
        st["x"] = _operands(case, seed)
        if kind == "transfer":
            x0, x1, y1, y2 = st["x"]
            st["y"] = [torch.empty_like(v) for v in (x1, y2, x0, y1)]
        else:
            st["y"] = torch.empty_like(st["x"][0])
        return st
    st["b"] = _rhs(case, seed)
    st["x"] = torch.empty_like(st["b"])
    if kind == "cold":
        st["params"] = mg.default_params(precision=PRECISION[case["precision"]], seed=int(seed) & 0xFFFFFFFF)
        return st
    params = mg.default_params(precision=PRECISION[case["precision"]], parallel=case["parallel"],
                               partial_tol=case["partial"])
    st["h"] = mg.mg_setup(U, Lx, Lt, M0, params=params)
    # the handle's first right-hand side builds the deflation space that later ones use
    b0 = _gauss((1, Lt, Lx, 2), seed, 21)
    mg.mg_solve(st["h"], b0, torch.empty_like(b0), 1, 1e-8)
    return st


def run(st):
    case = st["case"]
    kind = case["kind"]
    if kind == "wilson":
        prec = mg.MG_F64 if case["dtype"] == "f64" else mg.MG_F32
        mg.mg_wilson_apply(st["U"], case["Lx"], case["Lt"], M0, st["x"], st["y"], dagger=case["dagger"],
                           precision=prec)
        return st["y"]
    if kind == "stencil":
        prec = mg.MG_F64 if case["dtype"] == "f64" else mg.MG_F32
        mg.mg_apply(st["h"], case["level"], st["x"][0], st["y"], dagger=case["dagger"], precision=prec)
        return st["y"]
    if kind == "transfer":
        prec = mg.MG_F64 if case["dtype"] == "f64" else mg.MG_F32
        x0, x1, y1, y2 = st["x"]
        mg.mg_restrict(st["h"], 0, x0, st["y"][0], precision=prec)
        mg.mg_restrict(st["h"], 1, x1, st["y"][1], precision=prec)
        mg.mg_prolong(st["h"], 0, y1, st["y"][2], precision=prec)
        mg.mg_prolong(st["h"], 1, y2, st["y"][3], precision=prec)
        return st["y"]
    if kind == "block":
        mg.mg_apply_block(st["h"], case["level"], st["x"][0], st["y"], case["nrhs"],
                          precision=BLOCK_PRECISION[case["dtype"]])
        return st["y"]
    if kind == "cold":
        with mg.mg_setup(st["U"], case["Lx"], case["Lt"], M0, params=st["params"]) as h:
            mg.mg_solve(h, st["b"], st["x"], case["nrhs"], TOL)
        return st["x"]
    mg.mg_solve(st["h"], st["b"], st["x"], case["nrhs"], TOL)
    return st["x"]


def work(case):
    """Bytes and flops one pass cannot do without: inputs read once, outputs
    written once; of a solve the gauge field, right-hand sides and solutions, and
    one application of the fine operator to each."""
    sites = case["Lx"] * case["Lt"]
    kind = case["kind"]
    c = 16 if case.get("dtype") == "f64" else 8
    if kind == "wilson":
        return {"bytes": sites * 6 * c, "flops": sites * 70}
    if kind == "stencil":
        n = sites // 16 ** case["level"]
        entries = 576 + 4 * 192 if case["level"] == 1 else 5 * 576  # rank-4 hops on the intermediate grid
        return {"bytes": n * (entries + 48) * c, "flops": n * entries * 8}
    if kind == "block":
        n = sites // 16 ** case["level"]
        return {"bytes": n * (5 * 576 * 4 + case["nrhs"] * 48 * 8), "flops": n * 5 * 576 * 8 * case["nrhs"]}
    if kind == "transfer":
        n1, n2 = sites // 16, sites // 256
        q = n1 * 24 * 16 + n2 * 24 * 192  # prolongator entries, each read once by P^+ and by P
        return {"bytes": 2 * c * (q + 2 * sites + 24 * n1 + 24 * n1 + 24 * n2), "flops": 16 * q}
    return {"bytes": 16 * sites * (2 + 4 * case["nrhs"]), "flops": 70 * sites * case["nrhs"]}


# ------------------------------------------------------- 64-bit references ---


def _dirac(U, v, dagger=False):
    """D v (D^+ v) of spinors complex128[..., Lt, Lx, 2]."""
    sgn = -1.0 if dagger else 1.0
    ux, ut = U[..., 0], U[..., 1]
    p, q = v[..., 0], sgn * v[..., 1]
    Lt = U.shape[0]
    # antiperiodic in t: the forward hop out of the last row carries -1
    bc = torch.ones(Lt, 1, dtype=torch.float64, device=U.device)
    bc[-1] = -1.0
    utb = ut * bc
    hxp = ux * torch.roll(p - q, -1, -1)
    hxm = torch.roll(ux.conj() * (p + q), 1, -1)
    htp = utb * torch.roll(p + 1j * q, -1, -2)
    htm = torch.roll(utb.conj() * (p - 1j * q), 1, -2)
    a0 = hxp + hxm + htp + htm
    a1 = -hxp + hxm - 1j * htp + 1j * htm
    o0 = (M0 + 2) * p - 0.5 * a0
    o1 = sgn * ((M0 + 2) * q - 0.5 * a1)
    return torch.stack([o0, o1], -1)


def _blocks(v):
    """[..., Nt, Nx, dof] -> [..., Nt/4, Nx/4, 2, 16 dof/2]: the entries of each 4^2
    block and chirality, in the order of the prolongator's rows."""
    Nt, Nx, dof = v.shape[-3:]
    h = dof // 2
    w = v.reshape(v.shape[:-3] + (Nt // 4, 4, Nx // 4, 4, 2, h))
    d = w.dim()
    lead = list(range(d - 6))
    w = w.permute(lead + [d - 6, d - 4, d - 2, d - 5, d - 3, d - 1])
    return w.reshape(v.shape[:-3] + (Nt // 4, Nx // 4, 2, 16 * h))


def _unblocks(w, dof):
    bt, bx = w.shape[-4], w.shape[-3]
    h = dof // 2
    v = w.reshape(w.shape[:-4] + (bt, bx, 2, 4, 4, h))
    d = v.dim()
    lead = list(range(d - 6))
    v = v.permute(lead + [d - 6, d - 3, d - 5, d - 2, d - 4, d - 1])
    return v.reshape(w.shape[:-4] + (bt * 4, bx * 4, dof))


def _prolongator(nv):
    """Columns [bt, bx, 2, 12, 16 h], orthonormal per block and chirality (Gram-Schmidt,
    twice, in vector order)."""
    q = _blocks(nv)
    cols = []
    for j in range(NV):
        c = q[j]
        for _ in range(2):
            for p in cols:
                c = c - p * (p.conj() * c).sum(-1, keepdim=True)
            c = c / torch.linalg.vector_norm(c, dim=-1, keepdim=True)
        cols.append(c)
    return torch.stack(cols, -2)


def _restrict(P, v):
    out = torch.einsum("xycja,...xyca->...xycj", P.conj(), _blocks(v))
    return out.reshape(out.shape[:-2] + (24,))


def _prolong(P, v, dof):
    w = v.reshape(v.shape[:-1] + (2, NV))
    return _unblocks(torch.einsum("xycja,...xycj->...xyca", P, w), dof)


def _coarse_apply(U, P0, P1, level, x, dagger):
    """P^+ D P x on grid 1 or 2, one vector."""
    v = _prolong(P1, x, 24) if level == 2 else x
    v = _restrict(P0, _dirac(U, _prolong(P0, v, 2), dagger))
    return _restrict(P1, v) if level == 2 else v


def _solve(U, b):
    """D x = b by CG on D^+ D with refinement on the true residual, all right-hand sides at once."""
    x = torch.zeros_like(b)
    dims = (-3, -2, -1)

    def dot(u, v):
        return (u.conj() * v).real.sum(dims, keepdim=True)

    nb = torch.sqrt(dot(b, b))
    for _ in range(6):
        r0 = b - _dirac(U, x)
        if bool((torch.sqrt(dot(r0, r0)) <= 2e-14 * nb).all()):
            break
        r = _dirac(U, r0, True)
        e, p, rr = torch.zeros_like(b), r.clone(), dot(r, r)
        stop = 1e-12 * rr
        for it in range(20000):
            t = _dirac(U, p)
            alpha = rr / dot(t, t)
            e = e + alpha * p
            r = r - alpha * _dirac(U, t, True)
            new = dot(r, r)
            p = r + (new / rr) * p
            rr = new
            if it % 50 == 49 and bool((rr <= stop).all()):
                break
        x = x + e
    return x


def exact(case, seed):
    kind = case["kind"]
    U = _gauge(case["Lx"], case["Lt"], seed)
    if kind == "wilson":
        U = U.to(_cdtype(case["dtype"])).to(torch.complex128)
        return _dirac(U, _operands(case, seed)[0].to(torch.complex128), case["dagger"])
    if kind in ("solve", "cold"):
        if case["Lx"] * case["Lt"] * case["nrhs"] > 1 << 19:
            return None  # minutes of CG
        return _solve(U, _rhs(case, seed))
    nv0, nv1 = _null_vectors(case["Lx"], case["Lt"], seed)
    P0, P1 = _prolongator(nv0), _prolongator(nv1)
    x = [v.to(torch.complex128) for v in _operands(case, seed)]
    if kind == "transfer":
        return [_restrict(P0, x[0]), _restrict(P1, x[1]), _prolong(P0, x[2], 2), _prolong(P1, x[3], 24)]
    if kind == "block":
        return torch.stack([_coarse_apply(U, P0, P1, case["level"], v, False) for v in x[0]])
    return _coarse_apply(U, P0, P1, case["level"], x[0], case["dagger"])
