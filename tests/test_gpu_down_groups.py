"""GPU tests of the downward pass at the edges of its splits: one to seventeen
right-hand sides (groups of one to four, uneven last groups), rows of merges that
straddle warps, few rows (columns over a cluster) and many (one warp a row tile),
alone and in launches shared by several operators.

References: the oracle's solution for the first and the last column (1e-10, the
repository's bar) on small trees, and elsewhere every column against its own
one-column solve (1e-11: sums of the same products in another order)."""

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


def _operator(P, kind, p, L, f):
    pr = {"dtn2": W.elliptic_2d, "dtn3": W.elliptic_3d}.get(kind, lambda: W.helmholtz_bumps_2d(seed=1, k=6.0))()
    t = P.uniform_tree(pr.dim, L, pr.lo, pr.hi)
    x, _ = P.hps_nodes(t, p, p - 2)
    nl, ppl, nr = P.hps_sizes(t, p, p - 2)
    cf = pr.coeffs(x)
    a, b, c = cf["a"].reshape(nl, ppl), [v.reshape(nl, ppl) for v in cf["b"]], cf["c"].reshape(nl, ppl)
    d = lambda v: torch.from_numpy(np.ascontiguousarray(v)).cuda()  # noqa: E731
    h = P.hps_build(t, p, p - 2, P.HPS_ITI if kind == "iti" else P.HPS_DTN, a=d(a), b=[d(v) for v in b], c=d(c),
                    f=d(f(nl, ppl)), eta=pr.eta or 0.0)
    return pr, (a, b, c), h, nl, ppl, nr


@pytest.mark.parametrize("kind,p,L", [("dtn2", 5, 1), ("dtn2", 13, 3), ("dtn2", 9, 5), ("dtn3", 6, 1), ("dtn3", 7, 2),
                                      ("iti", 6, 1), ("iti", 13, 3), ("iti", 8, 5)])
@pytest.mark.parametrize("nrhs", [1, 2, 3, 4, 5, 7, 8, 17])
def test_columns(P, kind, p, L, nrhs):
    rng = np.random.default_rng(p + L)
    cx = kind == "iti"
    z = lambda *s: rng.standard_normal(s) + (1j * rng.standard_normal(s) if cx else 0)  # noqa: E731
    f = {}
    pr, (a, b, c), h, nl, ppl, nr = _operator(P, kind, p, L, lambda *s: f.setdefault(0, z(*s)))
    g = z(nrhs, nr)
    gd = torch.from_numpy(np.ascontiguousarray(g)).cuda()
    u = torch.empty((nrhs, nl, ppl), dtype=gd.dtype, device="cuda")
    P.hps_solve_batched(h, nrhs, gd, u)
    one = torch.empty((1, nl, ppl), dtype=gd.dtype, device="cuda")
    for k in range(nrhs):
        P.hps_solve(h, gd[k], one)
        assert float((one[0] - u[k]).abs().max()) <= 1e-11 * float(one.abs().max())
    if L <= 3 and kind != "dtn3":
        s = O.build(pr.dim, pr.kind, p, p - 2, L, pr.lo, pr.hi, a, b, c, f[0], eta=pr.eta)
        for k in {0, nrhs - 1}:
            uo = O.solve(s, g[k])
            assert np.abs(u[k].cpu().numpy() - uo).max() <= 1e-10 * np.abs(uo).max()
    # with an operator of another depth in shared launches
    _, _, h2, nl2, ppl2, nr2 = _operator(P, kind, p, max(L - 1, 0), z)
    g2 = torch.from_numpy(np.ascontiguousarray(z(1, nr2))).cuda()
    us = [torch.empty_like(u), torch.empty((1, nl2, ppl2), dtype=u.dtype, device="cuda")]
    ref = torch.empty_like(us[1])
    P.hps_solve_multi([h, h2], [gd, g2], us, nrhs=[nrhs, 1])
    P.hps_solve(h2, g2[0], ref)
    assert float((us[0] - u).abs().max()) <= 1e-11 * float(u.abs().max())
    assert float((us[1] - ref).abs().max()) <= 1e-11 * float(ref.abs().max())
