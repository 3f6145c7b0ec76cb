"""GPU tests of the leaf operators' assembly at its edges: one leaf spread over
many CTAs, more leaves than CTAs, the smallest and larger orders in both
dimensions, first-order terms, a zeroth-order term, trees with leaves of several
sizes.

Reference: the oracle's solution (1e-10, the repository's bar): an entry that is
missing, written twice or in a wrong place changes the solution by O(1)."""

import numpy as np
import pytest

import workloads as W
from oracle import hps as O

pytestmark = pytest.mark.gpu
torch = pytest.importorskip("torch")


@pytest.fixture(scope="module")
def P():
    if not torch.cuda.is_available():
        pytest.skip("no CUDA device")
    import paper_2503_17535_gb300 as P
    return P


CASES = [("dtn2", 4, 0), ("dtn2", 4, 3), ("dtn2", 17, 0), ("dtn2", 5, 5), ("dtn3", 4, 0), ("dtn3", 9, 0), ("dtn3", 5, 2),
         ("iti", 4, 0), ("iti", 4, 3), ("iti", 17, 1), ("iti", 5, 5)]


@pytest.mark.parametrize("kind,p,L", CASES, ids=["%s-p%d-L%d" % c for c in CASES])
def test_solution(P, kind, p, L):
    pr = {"dtn2": W.elliptic_2d, "dtn3": W.elliptic_3d}.get(kind, lambda: W.helmholtz_bumps_2d(seed=1, k=6.0))()
    t = P.uniform_tree(pr.dim, L, pr.lo, pr.hi)
    x, _ = P.hps_nodes(t, p, p - 2)
    nl, ppl, nr = P.hps_sizes(t, p, p - 2)
    cf = pr.coeffs(x)
    rng = np.random.default_rng(p + L)
    cx = kind == "iti"
    z = lambda *s: rng.standard_normal(s) + (1j * rng.standard_normal(s) if cx else 0)  # noqa: E731
    a, b, c = cf["a"].reshape(nl, ppl), [v.reshape(nl, ppl) for v in cf["b"]], cf["c"].reshape(nl, ppl)
    f, g = z(nl, ppl), z(nr)
    d = lambda v: torch.from_numpy(np.ascontiguousarray(v)).cuda()  # noqa: E731
    h = P.hps_build(t, p, p - 2, P.HPS_ITI if cx else P.HPS_DTN, a=d(a), b=[d(v) for v in b], c=d(c), f=d(f),
                    eta=pr.eta or 0.0)
    u = torch.empty((1, nl, ppl), dtype=d(f).dtype, device="cuda")
    P.hps_solve(h, d(g), u)
    uo = O.solve(O.build(pr.dim, pr.kind, p, p - 2, L, pr.lo, pr.hi, a, b, c, f, eta=pr.eta), g)
    assert np.abs(u[0].cpu().numpy() - uo).max() <= 1e-10 * np.abs(uo).max()
