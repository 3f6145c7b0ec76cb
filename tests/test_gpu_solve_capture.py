"""GPU tests of new-source solves on a stream that the caller captures.

The first solve with a new source forms the inverses of the factors' diagonal
blocks.  Recorded into a caller's graph it has formed nothing yet: a solve that
runs before the graph is launched, or after it is dropped, must form them
itself, and every launch of the graph must give the solution of the data that
are then behind its pointers.

Reference: the same solve of a second operator that was never captured.  The
same kernels run on the same data, so the results are equal, except where a
captured solve takes the blocked triangular solves (single factors beyond 2048
rows), which are as accurate: 1e-11, both are backward-stable solves."""

import numpy as np
import pytest

import workloads as W
from oracle import adaptive as ad

pytestmark = pytest.mark.gpu
torch = pytest.importorskip("torch")


@pytest.fixture(scope="module")
def P():
    if not torch.cuda.is_available():
        pytest.skip("no CUDA device")
    import paper_2503_17535_gb300 as P
    return P


def _operator(P, kind, p, L, lazy, seed):
    """(build(), g and f of a right-hand side from a seed, an output)."""
    pr = {"dtn2": W.elliptic_2d, "dtn3": W.elliptic_3d, "adaptive": W.elliptic_3d}.get(
        kind, lambda: W.helmholtz_bumps_2d(seed=1, k=6.0))()
    if kind == "adaptive":
        leaves = [(1, (i, j, k)) for i in range(2) for j in range(2) for k in range(2) if (i, j, k) != (0, 0, 0)]
        t = P.adaptive_tree(ad.sort_leaves(leaves + ad.children_of(1, (0, 0, 0))), pr.lo, pr.hi)
    else:
        t = P.uniform_tree(pr.dim, L, pr.lo, pr.hi)
    x, _ = P.hps_nodes(t, p, p - 2)
    nl, ppl, nr = P.hps_sizes(t, p, p - 2)
    cf = pr.coeffs(x)
    d = lambda v: torch.from_numpy(np.ascontiguousarray(v)).cuda()  # noqa: E731
    a, b, c = d(cf["a"].reshape(nl, ppl)), [d(v.reshape(nl, ppl)) for v in cf["b"]], d(cf["c"].reshape(nl, ppl))
    iti = kind == "iti"
    build = lambda: P.hps_build(t, p, p - 2, P.HPS_ITI if iti else P.HPS_DTN, a=a, b=b, c=c,  # noqa: E731
                                eta=pr.eta or 0.0, lazy_root=lazy)
    rng = np.random.default_rng(seed)

    def rhs():
        z = lambda *s: rng.standard_normal(s) + (1j * rng.standard_normal(s) if iti else 0)  # noqa: E731
        return d(z(nr)), d(z(nl, ppl))
    return build, rhs, lambda: torch.full((nl, ppl), float("nan"), dtype=torch.complex128 if iti else torch.float64, device="cuda")


CASES = [("dtn2", 9, 3, False), ("iti", 10, 3, False), ("iti", 10, 2, True), ("dtn3", 6, 2, False), ("dtn3", 6, 1, True),
         ("adaptive", 6, 0, False), ("dtn3", 9, 2, True)]


@pytest.mark.parametrize("kind,p,L,lazy", CASES, ids=["%s-p%d-L%d-%s" % (c[0], c[1], c[2], "lazy" if c[3] else "explicit")
                                                      for c in CASES])
def test_solves_around_a_callers_graph(P, kind, p, L, lazy):
    build, rhs, out = _operator(P, kind, p, L, lazy, 100 * p + L)
    (g, f), (g2, f2) = rhs(), rhs()
    blocked = (kind, p) == ("dtn3", 9)   # a root of 2352 rows
    same = lambda u, v: bool(((u - v).abs().max() <= (1e-11 if blocked else 0.0) * v.abs().max()))  # noqa: E731
    h = build()
    u, v = out(), out()
    P.hps_solve(h, g, u)   # the workspace
    torch.cuda.synchronize()
    dropped = torch.cuda.CUDAGraph()
    with torch.cuda.graph(dropped, capture_error_mode="thread_local"):
        P.hps_solve(h, g, u, f=f)
    del dropped
    P.hps_solve(h, g, v, f=f)
    ref = build()
    w, w2 = out(), out()
    P.hps_solve(ref, g, w, f=f)
    P.hps_solve(ref, g2, w2, f=f2)
    assert same(v, w)
    # a graph captured before any new-source solve, launched for three sources
    h = build()
    P.hps_solve(h, g, u)
    torch.cuda.synchronize()
    gin, fin = g.clone(), f.clone()
    graph = torch.cuda.CUDAGraph()
    with torch.cuda.graph(graph, capture_error_mode="thread_local"):
        P.hps_solve(h, gin, u, f=fin)
    for gk, fk, wk in ((g, f, w), (g2, f2, w2), (g, f, w)):
        gin.copy_(gk)
        fin.copy_(fk)
        u.fill_(float("nan"))
        graph.replay()
        assert same(u, wk)
    P.hps_solve(h, g2, v, f=f2)
    assert same(v, w2)
