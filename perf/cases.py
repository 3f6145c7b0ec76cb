"""The solver calls whose time matters, from the smallest to the largest.

A case is one call sequence of a user's program on one problem: build an
operator and solve with it, solve with an operator kept on the device, solve
with several kept operators at once, take a gradient, or form one dense
product.  The problems are the ones the benchmark and the tests use: 2D
Poisson, 2D and 3D variable-coefficient elliptic (Dirichlet-to-Neumann maps,
float64), 2D Helmholtz (impedance maps, complex128) and the 3D elliptic
operator on an octree refined around a sharp source.  Coefficients, sources and
boundary data are smooth fields drawn from the seed and evaluated on the GPU at
the solver's nodes.

listed()             the cases by name
draw(rng)            one more case of the same ranges
prepare(case, seed)  inputs and, where a program would keep one, the operator
run(state)           one pass through the public entry points
work(case)           bytes and flops one pass cannot do without
exact(case, seed)    the same outputs in plain 64-bit torch (below: a compact
                     leaf elimination, merge and downward pass over panels)
"""

from __future__ import annotations

import math
from functools import lru_cache

import numpy as np
import torch

import paper_2503_17535_gb300 as P
from paper_2503_17535_gb300.autograd import hps_solve_fn

DEV = "cuda"
DT = torch.float64
CDT = torch.complex128


# ---------------------------------------------------------------- cases ----

def listed():
    return [
        # a single small Dirichlet problem from scratch (16 leaves): a test, or
        # one patch of a larger program; launches and host calls are what counts
        {"name": "poisson2d_16_leaves", "op": "build_solve", "problem": "poisson2d", "depth": 2, "p": 8,
         "lazy": False, "newf": True},
        # the benchmark's step: Helmholtz operator on 4096 leaves, then a solve
        # with a new source
        {"name": "helmholtz2d_4096_leaves", "op": "build_solve", "problem": "helmholtz2d", "depth": 6, "p": 16,
         "k": 20.0, "lazy": True, "newf": True},
        # the 3D benchmark step: 512 leaves, one large dense root
        {"name": "elliptic3d_512_leaves", "op": "build_solve", "problem": "elliptic3d", "depth": 3, "p": 8,
         "lazy": True, "newf": True},
        # the adaptive 3D step: merges of many different sizes
        {"name": "adaptive3d_sharp_source", "op": "build_solve", "problem": "adaptive3d", "p": 8, "eps": 1e-4,
         "max_depth": 5, "width": 0.05, "cx": 0.21, "cy": -0.34, "cz": 0.13, "lazy": True, "newf": True},
        # a server's rebuild request with a new coefficient field: real 2D
        # operator of odd order with an explicit root, solved with the
        # build-time source
        {"name": "elliptic2d_rebuild_p13", "op": "build_solve", "problem": "elliptic2d", "depth": 5, "p": 13,
         "lazy": False, "newf": False},
        # leaves near resonance: the dense complex leaf factorisation
        {"name": "helmholtz2d_dense_leaves", "op": "build_solve", "problem": "helmholtz2d", "depth": 4, "p": 12,
         "k": 20.0, "lazy": False, "newf": False},
        # an apply-only request on a resident Helmholtz operator
        {"name": "apply_helmholtz2d", "op": "solve", "problem": "helmholtz2d", "depth": 6, "p": 16, "k": 20.0,
         "nrhs": 1, "lazy": False, "newf": False},
        # eight queued apply-only requests served as one batch (real operator)
        {"name": "apply_elliptic2d_batch8", "op": "solve", "problem": "elliptic2d", "depth": 6, "p": 16,
         "nrhs": 8, "lazy": False, "newf": False},
        # time stepping or an iteration over sources: new sources against a
        # resident operator, two at once
        {"name": "new_sources_helmholtz2d", "op": "solve", "problem": "helmholtz2d", "depth": 6, "p": 16,
         "k": 20.0, "nrhs": 2, "lazy": False, "newf": True},
        # apply-only requests of six operators of different kinds, depths and
        # orders in shared launches
        {"name": "serve_six_operators", "op": "multi",
         "operators": "iti:6:16,iti:3:12,iti:4:12,iti:6:12,dtn:6:16,dtn:5:8"},
        # one gradient of a misfit over the coefficient field (1024 leaves):
        # build, solve, adjoint solve, coefficient derivative
        {"name": "gradient_helmholtz2d", "op": "gradient", "problem": "helmholtz2d", "depth": 5, "p": 16,
         "k": 20.0},
        # the dense product alone, complex, ragged sizes
        {"name": "gemm_complex_ragged", "op": "gemm", "complex": True, "m": 1793, "n": 1211, "k": 449, "batch": 3},
    ]


def draw(rng):
    def log_int(lo, hi):
        return int(round(math.exp(rng.uniform(math.log(lo), math.log(hi)))))

    op = rng.choice(["build_solve", "build_solve", "build_solve", "solve", "solve", "multi", "gradient", "gemm"])
    if op == "gemm":
        c = rng.random() < 0.5
        return {"op": op, "complex": c, "m": log_int(17, 2500), "n": log_int(17, 2500), "k": log_int(17, 1200),
                "batch": log_int(1, 6)}
    if op == "multi":
        n = rng.randint(2, 6)
        kinds = [(rng.choice(["iti", "dtn"]), rng.randint(3, 6), rng.choice([8, 12, 16])) for _ in range(n)]
        return {"op": op, "operators": ",".join("%s:%d:%d" % k for k in kinds)}
    if op == "gradient":
        prob = rng.choice(["helmholtz2d", "elliptic2d"])
        case = {"op": op, "problem": prob, "depth": rng.randint(2, 5), "p": rng.randint(8, 16)}
        if prob == "helmholtz2d":
            case["k"] = round(rng.uniform(5.0, 30.0), 3)
        return case
    prob = rng.choice(["poisson2d", "elliptic2d", "helmholtz2d", "helmholtz2d", "elliptic3d", "adaptive3d"])
    case = {"op": op, "problem": prob, "lazy": rng.random() < 0.5, "newf": rng.random() < 0.5}
    if prob == "adaptive3d":
        case.update(p=rng.randint(6, 8), eps=1e-4, max_depth=rng.randint(3, 5), width=round(rng.uniform(0.05, 0.09), 4),
                    cx=round(rng.uniform(-0.5, 0.5), 3), cy=round(rng.uniform(-0.5, 0.5), 3),
                    cz=round(rng.uniform(-0.5, 0.5), 3))
    elif prob == "elliptic3d":
        case["depth"] = rng.randint(1, 3)
        case["p"] = rng.randint(5, 8) if case["depth"] == 3 else rng.randint(5, 10)
    else:
        case["depth"] = rng.randint(1, 6)
        case["p"] = rng.randint(6, 16)
        if prob == "helmholtz2d":
            case["k"] = round(rng.uniform(5.0, 30.0), 3)
    if op == "solve":
        case["nrhs"] = 1 if prob == "adaptive3d" else log_int(1, 8)
    return case


# --------------------------------------------------------------- inputs ----

def _is_iti(problem):
    return problem == "helmholtz2d"


def _dim(problem):
    return 3 if problem.endswith("3d") else 2


@lru_cache(maxsize=8)
def _octree(p, eps, max_depth, width, cx, cy, cz):
    def sharp(x):
        return np.exp(-((x - np.array([cx, cy, cz])) ** 2).sum(axis=1) / (2 * width ** 2))
    return P.hps_refine((-1.0,) * 3, (1.0,) * 3, p, eps, 2, max_depth, [sharp])


def _tree(case):
    """(tree, leaves or None)."""
    if case["problem"] == "adaptive3d":
        leaves = _octree(case["p"], case["eps"], case["max_depth"], case["width"], case["cx"], case["cy"], case["cz"])
        return P.adaptive_tree(leaves), leaves
    return P.uniform_tree(_dim(case["problem"]), case["depth"]), None


@lru_cache(maxsize=4)
def _uniform_nodes(dim, depth, p):
    """Leaf and boundary nodes of a uniform tree on the device, laid out once."""
    x, xb = P.hps_nodes(P.uniform_tree(dim, depth), p, p - 2)
    return torch.from_numpy(x).to(DEV), torch.from_numpy(xb).to(DEV)


def _nodes(case, tree):
    if case["problem"] != "adaptive3d":
        return _uniform_nodes(_dim(case["problem"]), case["depth"], case["p"])
    x, xb = P.hps_nodes(tree, case["p"], case["p"] - 2)
    return torch.from_numpy(x).to(DEV), torch.from_numpy(xb).to(DEV)


def _waves(x, rng, n, kmax):
    """A smooth field: n seeded sine waves, amplitudes adding up to 1."""
    k = rng.uniform(-kmax, kmax, (n, x.shape[1]))
    ph, am = rng.uniform(0, 2 * np.pi, n), rng.uniform(0.2, 1.0, n)
    arg = x @ torch.from_numpy(k.T.copy()).to(DEV) + torch.from_numpy(ph).to(DEV)
    return torch.sin(arg) @ torch.from_numpy(am / am.sum()).to(DEV)


def _coefficients(case, x, rng):
    """{"a", "b", "c"} at the nodes (None: the library's constants)."""
    prob = case["problem"]
    if prob == "poisson2d":
        return {"a": None, "b": None, "c": None}
    if prob == "helmholtz2d":
        z = torch.from_numpy(rng.uniform(-0.8, 0.8, (4, 2))).to(DEV)
        n = sum(0.5 * torch.exp(-((x - z[i]) ** 2).sum(1) / (2 * 0.1 ** 2)) for i in range(4))
        return {"a": None, "b": None, "c": case["k"] ** 2 * (1.0 - n)}
    # div(a grad u) + c u with a in [0.5, 1.5], expanded: b = grad a
    dim = x.shape[1]
    km, ph, al = rng.uniform(-3, 3, (8, dim)), rng.uniform(0, 2 * np.pi, 8), rng.uniform(-1, 1, 8)
    al = 0.5 * al / np.abs(al).sum()
    kt, at = torch.from_numpy(km).to(DEV), torch.from_numpy(al).to(DEV)
    arg = x @ kt.T + torch.from_numpy(ph).to(DEV)
    ga = (torch.cos(arg) * at) @ kt
    return {"a": 1.0 + torch.sin(arg) @ at, "b": [ga[:, j].contiguous() for j in range(dim)],
            "c": 0.5 + 0.5 * _waves(x, rng, 2, 2.0)}


def _source(case, x, rng):
    if case["problem"] == "adaptive3d":
        z = torch.tensor([case["cx"], case["cy"], case["cz"]], dtype=DT, device=DEV)
        f = rng.uniform(0.5, 2.0) * torch.exp(-((x - z) ** 2).sum(1) / (2 * case["width"] ** 2)) + 0.1 * _waves(x, rng, 2, 2.0)
    else:
        z = torch.from_numpy(rng.uniform(-0.8, 0.8, x.shape[1])).to(DEV)
        f = torch.exp(-((x - z) ** 2).sum(1) / (2 * 0.1 ** 2)) + 0.2 * _waves(x, rng, 3, 4.0)
    if _is_iti(case["problem"]):
        f = torch.complex(f, 0.3 * _waves(x, rng, 3, 4.0))
    return f


def _boundary(case, xb, rng):
    if not _is_iti(case["problem"]):
        return _waves(xb, rng, 4, 4.0)
    # incoming impedance of a plane wave
    th, k = rng.uniform(0, 2 * np.pi), case["k"]
    d = torch.tensor([math.cos(th), math.sin(th)], dtype=DT, device=DEV)
    nrm = torch.where(xb.abs() >= 1.0 - 1e-12, torch.sign(xb), torch.zeros_like(xb))
    w = torch.exp(1j * k * (xb @ d))
    return 1j * k * (nrm @ d) * w + 1j * k * w


def _inputs(case, seed):
    """Everything a program has in hand before the call, from the seed."""
    rng = np.random.default_rng(seed)
    if case["op"] == "gemm":
        g = torch.Generator(device=DEV).manual_seed(int(seed))
        dt = CDT if case["complex"] else DT
        m, n, k, b = case["m"], case["n"], case["k"], case["batch"]
        mk = lambda *s: torch.randn(*s, dtype=dt, device=DEV, generator=g)  # noqa: E731
        return {"A": mk(b, k, m), "B": mk(b, n, k), "C": mk(b, n, m)}
    tree, leaves = _tree(case)
    p = case["p"]
    x, xb = _nodes(case, tree)
    npl = p ** _dim(case["problem"])
    nl, nr = x.shape[0] // npl, case.get("nrhs", 1)
    co = _coefficients(case, x, rng)
    s = {"tree": tree, "leaves": leaves, "p": p, "kind": P.HPS_ITI if _is_iti(case["problem"]) else P.HPS_DTN,
         "eta": float(case.get("k", 0.0)), "co": co, "f0": _source(case, x, rng).reshape(nl, npl),
         "g": torch.stack([_boundary(case, xb, rng) for _ in range(nr)])}
    s["f"] = torch.stack([_source(case, x, rng).reshape(nl, npl) for _ in range(nr)]) if case.get("newf") else None
    if case["op"] == "gradient":
        s["obs"] = _source(case, x, rng).reshape(nl, npl)
        if co["c"] is None:
            co["c"] = torch.zeros(nl * npl, dtype=DT, device=DEV)
        co["c"] = co["c"].reshape(nl, npl)
    s["u"] = torch.empty((nr, nl, npl), dtype=CDT if s["kind"] == P.HPS_ITI else DT, device=DEV)
    return s


def _build(s, lazy):
    co = s["co"]
    return P.hps_build(s["tree"], s["p"], s["p"] - 2, s["kind"], a=co["a"], b=co["b"], c=co["c"], f=s["f0"],
                       eta=s["eta"], lazy_root=lazy)


def _operators(case):
    """The single-operator cases a "multi" case consists of."""
    out = []
    for word in case["operators"].split(","):
        kind, depth, p = word.split(":")
        out.append({"op": "solve", "problem": "helmholtz2d" if kind == "iti" else "elliptic2d", "depth": int(depth),
                    "p": int(p), "k": 20.0, "nrhs": 1, "lazy": False, "newf": False})
    return out


def prepare(case, seed):
    if case["op"] == "multi":
        parts = [prepare(c, 1000 * int(seed) + i) for i, c in enumerate(_operators(case))]
        return {"op": "multi", "parts": parts}
    s = _inputs(case, seed)
    s["op"] = case["op"]
    s["lazy"] = bool(case.get("lazy", False))
    if case["op"] == "solve":
        s["h"] = _build(s, s["lazy"])
    return s


def run(s):
    op = s["op"]
    if op == "build_solve":
        h = _build(s, s["lazy"])
        P.hps_solve(h, s["g"], s["u"], f=s["f"])
        P.hps_free(h)
        return s["u"]
    if op == "solve":
        P.hps_solve_batched(s["h"], s["u"].shape[0], s["g"], s["u"], f=s["f"])
        return s["u"]
    if op == "multi":
        parts = s["parts"]
        P.hps_solve_multi([t["h"] for t in parts], [t["g"] for t in parts], [t["u"] for t in parts])
        return [t["u"] for t in parts]
    if op == "gradient":
        co = s["co"]
        c, g, f = (v.detach().requires_grad_() for v in (co["c"], s["g"][0], s["f0"]))
        u = hps_solve_fn(c, g, f, s["tree"], s["p"], s["kind"], a=co["a"], b=co["b"], eta=s["eta"])
        r = u - s["obs"]
        J = (r * r.conj()).real.sum()
        gc, gg, gf = torch.autograd.grad(J, (c, g, f))
        return {"u": u.detach(), "grad_c": gc, "grad_g": gg, "grad_f": gf}
    C = s["C"].clone()
    P.hps_gemm(s["A"], s["B"], C, alpha=-1.0, beta=1.0)
    return C


# ----------------------------------------------------------------- work ----

def _level_sizes(dim, depth, p, iti):
    """[(merges, n_int, n_ext, unknowns factored)] from the leaves up."""
    q = p - 2
    out = []
    for m in range(depth):
        side = (2 ** m) * q if dim == 2 else (4 ** m) * q * q    # points of one child face
        ni = (4 if dim == 2 else 12) * side
        ni, nlu = (2 * ni, ni) if iti else (ni, ni)
        out.append((2 ** (dim * (depth - 1 - m)), ni, (8 if dim == 2 else 24) * side, nlu))
    return out


def work(case):
    if case["op"] == "gemm":
        m, n, k, b = case["m"], case["n"], case["k"], case["batch"]
        w, f = (16, 8) if case["complex"] else (8, 2)
        return {"bytes": float(w * b * (m * k + k * n + 2 * m * n)), "flops": float(f) * m * n * k * b}
    if case["op"] == "multi":
        ws = [work(c) for c in _operators(case)]
        return {k: sum(w[k] for w in ws) for k in ("bytes", "flops")}
    prob, p = case["problem"], case["p"]
    dim, iti = _dim(prob), _is_iti(prob)
    es, fm = (16, 8.0) if iti else (8, 2.0)
    npl, q = p ** dim, p - 2
    nb = 4 * q if dim == 2 else 6 * q * q
    ni = (p - 2) ** dim
    nr = case.get("nrhs", 1)
    if prob == "adaptive3d":
        nl = len(_octree(p, case["eps"], case["max_depth"], case["width"], case["cx"], case["cy"], case["cz"]))
        # merges about as large as those of a uniform tree of as many leaves
        depth = max(1, round(math.log(nl, 8)))
        levels = [(max(1, nl * n // 8 ** depth), a, b, c) for n, a, b, c in _level_sizes(3, depth, p, False)]
    else:
        nl = 2 ** (dim * case["depth"])
        levels = _level_sizes(dim, case["depth"], p, iti)
    lazy = bool(case.get("lazy", False))
    ncoef = 0 if prob == "poisson2d" else 1 if iti else dim + 2
    vec = nl * npl
    # leaf: LU of the interior block and nb + 1 right-hand sides (real), the
    # boundary Schur complement of an impedance leaf, and T
    leaf = 2.0 / 3.0 * ni ** 3 + 2.0 * ni * ni * (nb + 1) + 2.0 * nb * ni * (nb + 1)
    if iti:
        no = 4 * (p - 1)
        leaf = 2.0 / 3.0 * ni ** 3 + 2.0 * ni * ni * no + 2.0 * no * no * ni + 8.0 / 3.0 * no ** 3 \
            + 8.0 * no * no * (nb + 1) + 4.0 * ni * no * (nb + 1) + 4.0 * nb * npl * (nb + 1)
    build = nl * leaf
    apply_el, up_el = float(nl * npl * (nb + 1)), float(nl * (ni * ni + nb * ni))
    for t, (nm, mi, me, nlu) in enumerate(levels):
        top = t == len(levels) - 1
        lu = fm / 3.0 * nlu ** 3
        rhs = 0.0 if (top and lazy) else fm * nlu * nlu * (me + 1) * (2.0 if iti else 1.0)
        schur = 0.0 if top else fm * me * (me + 1) * mi / (2.0 if dim == 2 else 4.0)
        build += nm * (lu + rhs + schur)
        apply_el += nm * mi * (me + 1)
        up_el += nm * (nlu * nlu + (0 if top else me * mi / 4.0))
    newf = bool(case.get("newf"))
    io = es * vec * nr * (2 if newf else 1)
    if case["op"] == "solve":
        el = apply_el + (up_el if newf else 0.0)
        return {"bytes": es * el + io, "flops": fm * el * nr}
    if case["op"] == "gradient":
        return {"bytes": 8.0 * vec * (ncoef + 1) + es * vec * 4, "flops": build + 2 * fm * (apply_el + up_el)}
    solve = fm * (apply_el + (up_el if newf else 0.0))
    return {"bytes": 8.0 * vec * ncoef + es * vec * (3 if newf else 2), "flops": build + solve}


# ---------------------------------------------------------------- exact ----
#
# The discretisation once more in plain torch: leaf collocation on p
# Chebyshev points a side, boundary maps on q = p - 2 Gauss points a panel,
# merges by eliminating the siblings' shared panels, the downward pass.  A
# node's boundary is a list of panels (face, level, position); where a shared
# panel has four finer ones on one side, those enter through the coarse
# panel's interpolant and leave through its L2 projection.

FACES = {2: [(1, 0), (0, 1), (1, 1), (0, 0)], 3: [(a, s) for a in range(3) for s in (0, 1)]}


def _t(v):
    return torch.from_numpy(np.ascontiguousarray(v)).to(DEV)


def _cheb(p):
    return -np.cos(np.pi * np.arange(p) / (p - 1))


def _bary(x):
    d = x[:, None] - x[None, :] + np.eye(len(x))
    w = 1.0 / d.prod(axis=1)
    return w / np.abs(w).max()


def _diff(x):
    w, n = _bary(x), len(x)
    D = (w[None, :] / w[:, None]) / (x[:, None] - x[None, :] + np.eye(n))
    D[np.arange(n), np.arange(n)] = 0.0
    D[np.arange(n), np.arange(n)] = -D.sum(axis=1)
    return D


def _interp(src, dst):
    w, d = _bary(src), dst[:, None] - src[None, :]
    hit = d == 0.0
    r = w / np.where(hit, 1.0, d)
    M = r / r.sum(axis=1, keepdims=True)
    rows = hit.any(axis=1)
    M[rows] = hit[rows]
    return M


def _kron(ms):
    """Operator of a tensor grid whose first axis runs fastest."""
    out = np.ones((1, 1))
    for m in ms:
        out = np.kron(m, out)
    return out


def _leaf_maps(dim, p, iti, hl, co, f, eta):
    """Batched leaf stage: u = Y g + v, outgoing data = T g + h.  hl: leaf
    sides (batch), co: a, b, c (batch, p^dim) or None, f (batch, p^dim)."""
    q, npl = p - 2, p ** dim
    x, xg = _cheb(p), np.polynomial.legendre.leggauss(p - 2)[0]
    D, I = _diff(x), np.eye(p)
    Ds = [_kron([D if k == a else I for k in range(dim)]) for a in range(dim)]
    grid = np.indices((p,) * dim).reshape(dim, -1)[::-1]          # grid[a]: index along axis a, first axis fastest
    inner = np.all((grid > 0) & (grid < p - 1), axis=0)
    Ii, Ie = np.nonzero(inner)[0], np.nonzero(~inner)[0]
    faces = [np.nonzero(grid[a] == (p - 1 if s else 0))[0] for a, s in FACES[dim]]   # lower tangential axis fastest
    GC, CG = _kron([_interp(xg, x)] * (dim - 1)), _kron([_interp(x, xg)] * (dim - 1))
    n0, nb = q ** (dim - 1), 2 * dim * q ** (dim - 1)
    s = (2.0 / hl)[:, None, None]
    a, b, c = co
    L = sum(_t(M @ M) for M in Ds) * s * s
    if a is not None:
        L = a[:, :, None] * L
    if b is not None:
        L = L + sum(b[k][:, :, None] * _t(Ds[k]) for k in range(dim)) * s
    if c is not None:
        L = L + torch.diag_embed(c)
    B = hl.shape[0]
    if L.shape[0] == 1 and B > 1:
        L = L.expand(B, npl, npl)
    ti, te = torch.from_numpy(Ii).to(DEV), torch.from_numpy(Ie).to(DEV)
    if not iti:
        Pm, Q = np.zeros((npl, nb)), np.zeros((nb, npl))
        times = sum(np.isin(np.arange(npl), nd).astype(float) for nd in faces)
        for k, (nd, (ax, sd)) in enumerate(zip(faces, FACES[dim])):
            Pm[nd, k * n0:(k + 1) * n0] += GC / times[nd][:, None]
            Q[k * n0:(k + 1) * n0] = CG @ ((1.0 if sd else -1.0) * Ds[ax][nd])
        Pe = _t(Pm[Ie])
        Li = L[:, ti]
        X = torch.linalg.solve(Li[:, :, ti], torch.cat([Li[:, :, te] @ Pe, -f[:, ti, None].to(L.dtype)], 2))
        YV = torch.zeros((B, npl, nb + 1), dtype=DT, device=DEV).index_copy(1, ti, -X)
        YV = YV + torch.cat([_t(Pm), torch.zeros((npl, 1), dtype=DT, device=DEV)], 1)
        TH = (_t(Q) * s) @ YV
    else:
        own = [np.arange(p - 1), np.arange(p - 1), np.arange(1, p), np.arange(1, p)]
        no = 4 * (p - 1)
        Gd, Gu, Pm = np.zeros((no, npl)), np.zeros((no, npl)), np.zeros((no, nb))
        Hd, Hu, r = np.zeros((nb, npl)), np.zeros((nb, npl)), 0
        for k, (nd, (ax, sd)) in enumerate(zip(faces, FACES[2])):
            sg, ow = (1.0 if sd else -1.0), own[k]
            Gd[r:r + p - 1] = sg * Ds[ax][nd[ow]]
            Gu[np.arange(r, r + p - 1), nd[ow]] = 1.0
            Pm[r:r + p - 1, k * q:(k + 1) * q] = GC[ow]
            Hd[k * q:(k + 1) * q] = CG @ (sg * Ds[ax][nd])
            Hu[k * q:(k + 1) * q][:, nd] = CG
            r += p - 1
        G = _t(Gd) * s + 1j * eta * _t(Gu)
        Bm = torch.cat([G.expand(B, no, npl), L[:, ti].to(CDT)], 1)
        top = torch.cat([_t(Pm).to(CDT), torch.zeros((no, 1), dtype=CDT, device=DEV)], 1).expand(B, no, nb + 1)
        low = torch.cat([torch.zeros((B, len(Ii), nb), dtype=CDT, device=DEV), f[:, ti, None].to(CDT)], 2)
        YV = torch.linalg.solve(Bm, torch.cat([top, low], 1))
        TH = (_t(Hd) * s - 1j * eta * _t(Hu)) @ YV
    return YV, TH


@lru_cache(maxsize=None)
def _panel_maps(q):
    """Coarse 3D panel data at its four finer panels, and the L2 projection back."""
    xc, wc = np.polynomial.legendre.leggauss(q)
    c2f = _interp(xc, np.concatenate([(xc - 1) / 2, (xc + 1) / 2]))
    f2c = (c2f * np.concatenate([wc, wc])[:, None] / 2).T / wc[:, None]
    cut = [slice(0, q), slice(q, 2 * q)]
    C2F = [_kron([c2f[cut[k & 1]], c2f[cut[k >> 1]]]) for k in range(4)]
    F2C = [_kron([f2c[:, cut[k & 1]], f2c[:, cut[k >> 1]]]) for k in range(4)]
    return np.concatenate(C2F, 0), np.concatenate(F2C, 1)


def _split_panel(pan):
    lev, pos = pan
    return [(lev + 1, tuple(2 * v + ((k >> i) & 1) for i, v in enumerate(pos))) for k in range(2 ** len(pos))]


def _leaf_panels(dim, level, idx):
    return [[(level, tuple(idx[t] for t in range(dim) if t != ax))] for ax, _ in FACES[dim]]


def _join(dim, kids, n0, iti):
    """Faces of the parent and, per child, (R, E, ext, var, eq): its data in
    merge order is E from / R onto the interface panels (None: unchanged),
    ext / var / eq the parent's exterior, unknown and equation numbers (-1)."""
    faces = []
    for fc, (ax, sd) in enumerate(FACES[dim]):
        tang = [t for t in range(dim) if t != ax]
        lst = []
        for k in range(2 ** (dim - 1)):
            c = (sd << ax) + sum(((k >> i) & 1) << t for i, t in enumerate(tang))
            lst += kids[c][fc]
        faces.append(lst)
    ext_no, n = {}, 0
    for fc, lst in enumerate(faces):
        for pan in lst:
            ext_no[(fc, pan)] = n
            n += n0
    n_ext = n
    fno = {v: k for k, v in enumerate(FACES[dim])}
    shared, n = {}, 0                    # (axis, panel, low child's face set) -> number
    for ax in range(dim):
        for c in range(2 ** dim):
            if (c >> ax) & 1:
                continue
            lo, hi = kids[c][fno[(ax, 1)]], kids[c | (1 << ax)][fno[(ax, 0)]]
            los, his = set(lo), set(hi)
            up = {(p[0] - 1, tuple(v >> 1 for v in p[1])) for p in los ^ his}
            coarse = [p for p in lo if p in his or p in up] + [p for p in hi if p not in los and p in up]
            for pan in coarse:
                shared[(ax, c, pan)] = n
                n += n0
    n_int = n * (2 if iti else 1)
    plans = []
    for c, kid in enumerate(kids):
        ext, var, eq, Rr, off = [], [], [], [], 0
        mixed = False
        for fc, (ax, sd) in enumerate(FACES[dim]):
            where = {}
            for pan in kid[fc]:
                where[pan] = off
                off += n0
            if sd == ((c >> ax) & 1):
                for pan in kid[fc]:
                    Rr.append([where[pan]])
                    ext += range(ext_no[(fc, pan)], ext_no[(fc, pan)] + n0)
                    var += [-1] * n0
                    eq += [-1] * n0
                continue
            low = c if sd == 1 else c ^ (1 << ax)
            for (ax2, c2, pan), base in shared.items():
                if ax2 != ax or c2 != low:
                    continue
                if pan in where:
                    Rr.append([where[pan]])
                else:
                    mixed = True
                    Rr.append([where[p] for p in _split_panel(pan)])
                ext += [-1] * n0
                if iti:                  # own incoming data; the row belongs to the neighbour's
                    mine, his = (base, base + n) if sd == 1 else (base + n, base)
                    var += range(mine, mine + n0)
                    eq += range(his, his + n0)
                else:
                    var += range(base, base + n0)
                    eq += range(base, base + n0)
        npr = len(ext)
        if mixed:
            C2F, F2C = _panel_maps(round(math.sqrt(n0)))
            R, E = np.zeros((npr, off)), np.zeros((off, npr))
            for k, src in enumerate(Rr):
                rows = slice(k * n0, (k + 1) * n0)
                for j, o in enumerate(src):
                    fine = slice(j * n0, (j + 1) * n0)
                    R[rows, o:o + n0] = np.eye(n0) if len(src) == 1 else F2C[:, fine]
                    E[o:o + n0, rows] = np.eye(n0) if len(src) == 1 else C2F[fine]
            R, E = _t(R), _t(E)
        else:
            R = E = torch.from_numpy(np.concatenate([np.arange(o[0], o[0] + n0) for o in Rr])).to(DEV)
        ext, var, eq = (np.array(v) for v in (ext, var, eq))
        e, i = np.nonzero(ext >= 0)[0], np.nonzero(ext < 0)[0]
        ix = [torch.from_numpy(v).to(DEV) for v in (e, i, ext[e], var[i], eq[i])]
        plans.append((mixed, R, E, ix))
    return faces, n_ext, n_int, plans


def _merge(TH, join, iti, top):
    """TH: per child [T | h], batched over merges."""
    _, ne, ni, plans = join
    B, dt = TH[0].shape[0], TH[0].dtype
    z = lambda m, n: torch.zeros((B, m, n), dtype=dt, device=DEV)  # noqa: E731
    D, C = z(ni, ni), z(ni, ne + 1)
    if iti:
        D = D + torch.eye(ni, dtype=dt, device=DEV)
    parts = []
    for th, (mixed, R, E, (e, i, ext, var, eq)) in zip(TH, plans):
        n = th.shape[1]
        T, h = th[:, :, :n], th[:, :, n:]
        if mixed:
            T, h = R @ T @ E, R @ h
        else:
            T, h = T[:, R][:, :, R], h[:, R]
        D = _add(D, eq, var, T[:, i][:, :, i])
        C = _add(C, eq, ext, T[:, i][:, :, e])
        C = _add(C, eq, torch.full((1,), ne, device=DEV), h[:, i])
        parts.append((T, h))
    if top:
        return (D, C), None
    X = torch.linalg.solve(D, C)
    out = z(ne, ne + 1)
    last = torch.full((1,), ne, device=DEV)
    for (T, h), (_, _, _, (e, i, ext, var, eq)) in zip(parts, plans):
        out = _add(out, ext, ext, T[:, e][:, :, e])
        out = _add(out, ext, last, h[:, e])
        out = _add(out, ext, torch.arange(ne + 1, device=DEV), -(T[:, e][:, :, i] @ X[:, var]))
    return X, out


def _add(M, r, c, v):
    b = torch.arange(M.shape[0], device=DEV)
    return M.index_put((b[:, None, None], r[None, :, None], c[None, None, :]), v, accumulate=True)


def _down(g, gint, join):
    """Boundary data of the children from the parent's g (batch, n_ext)."""
    out = []
    for mixed, R, E, (e, i, ext, var, eq) in join[3]:
        v = torch.zeros((g.shape[0], len(e) + len(i)), dtype=g.dtype, device=DEV)
        v = v.index_copy(1, e, g[:, ext]).index_copy(1, i, gint[:, var])
        out.append(v @ E.T.to(v.dtype) if mixed else torch.zeros_like(v).index_copy(1, E, v))
    return out


def _solution(case, s, c, g, f):
    """u (leaves, nodes) for one right-hand side."""
    dim, iti, p = _dim(case["problem"]), _is_iti(case["problem"]), case["p"]
    npl, n0 = p ** dim, (p - 2) ** (dim - 1)
    r = lambda v: None if v is None else v.reshape(-1, npl)  # noqa: E731
    co = (r(s["co"]["a"]), None if s["co"]["b"] is None else [r(v) for v in s["co"]["b"]], r(c))
    f = f.reshape(-1, npl)
    nl = f.shape[0]
    if s["leaves"] is None:
        L = case["depth"]
        hl = torch.full((nl,), 2.0 / 2 ** L, dtype=DT, device=DEV)
        YV, TH = _leaf_maps(dim, p, iti, hl, co, f, s["eta"])
        faces = [_leaf_panels(dim, L, [(k >> t) & 1 for t in range(dim)]) for k in range(2 ** dim)]
        joins, Xs = [], []
        for m in range(L):
            join = _join(dim, faces, n0, iti)
            nch, top = 2 ** dim, m == L - 1
            TH = TH.reshape(-1, nch, *TH.shape[1:])
            X, TH = _merge([TH[:, k] for k in range(nch)], join, iti, top)
            joins.append(join)
            Xs.append(X)
            if not top:   # the same structure for every sibling: shift the panels
                lev = L - 1 - m
                faces = [[[(a, tuple(v + (((k >> t) & 1) << (a - lev)) for v, t in zip(b, [t for t in range(dim) if t != ax])))
                           for a, b in lst] for lst, (ax, _) in zip(join[0], FACES[dim])] for k in range(2 ** dim)]
        gv = g[None]
        for m in range(L - 1, -1, -1):
            if m == L - 1:
                D, C = Xs[m]
                gi = -torch.linalg.solve(D, C[:, :, :-1] @ gv[:, :, None] + C[:, :, -1:])[:, :, 0]
            else:
                gi = -(Xs[m][:, :, :-1] @ gv[:, :, None] + Xs[m][:, :, -1:])[:, :, 0]
            gv = torch.stack(_down(gv, gi, joins[m]), 1).reshape(-1, joins[m][3][0][2].shape[0])
        return (YV[:, :, :-1] @ gv[:, :, None] + YV[:, :, -1:])[:, :, 0]
    leaves = s["leaves"]
    hl = torch.tensor([2.0 / 2 ** lv for lv, _ in leaves], dtype=DT, device=DEV)
    YV, TH = _leaf_maps(3, p, False, hl, co, f, 0.0)
    row = {lf: k for k, lf in enumerate(leaves)}
    kids_of = lambda lv, ix: [(lv + 1, tuple(2 * ix[t] + ((k >> t) & 1) for t in range(3))) for k in range(8)]  # noqa: E731
    kept, gl = {}, {}

    def up(node):
        if node in row:
            return _leaf_panels(3, *node), TH[row[node]][None]
        got = [up(k) for k in kids_of(*node)]
        join = _join(3, [v[0] for v in got], n0, False)
        X, out = _merge([v[1] for v in got], join, False, node[0] == 0)
        kept[node] = (join, X)
        return join[0], out

    def down(node, gv):
        if node in row:
            gl[row[node]] = gv[0]
            return
        join, X = kept[node]
        if node[0] == 0:
            gi = -torch.linalg.solve(X[0], X[1][:, :, :-1] @ gv[:, :, None] + X[1][:, :, -1:])[:, :, 0]
        else:
            gi = -(X[:, :, :-1] @ gv[:, :, None] + X[:, :, -1:])[:, :, 0]
        for k, v in zip(kids_of(*node), _down(gv, gi, join)):
            down(k, v)

    up((0, (0, 0, 0)))
    down((0, (0, 0, 0)), g[None])
    gv = torch.stack([gl[k] for k in range(nl)])
    return (YV[:, :, :-1] @ gv[:, :, None] + YV[:, :, -1:])[:, :, 0]


def exact(case, seed):
    if case["op"] == "gemm":
        s = _inputs(case, seed)
        return s["C"] - torch.bmm(s["B"], s["A"])      # columns contiguous: C^T = B^T A^T
    if case["op"] == "multi":
        return [exact(c, 1000 * int(seed) + i) for i, c in enumerate(_operators(case))]
    s = _inputs(case, seed)
    c = s["co"]["c"]
    if case["op"] == "gradient":
        c, g, f = (v.detach().requires_grad_() for v in (c, s["g"][0], s["f0"]))
        u = _solution(case, s, c, g, f)
        r = u - s["obs"]
        gc, gg, gf = torch.autograd.grad((r * r.conj()).real.sum(), (c, g, f))
        return {"u": u.detach(), "grad_c": gc, "grad_g": gg, "grad_f": gf}
    with torch.no_grad():
        return torch.stack([_solution(case, s, c, s["g"][k], s["f0"] if s["f"] is None else s["f"][k])
                            for k in range(s["g"].shape[0])])
