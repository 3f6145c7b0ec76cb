"""GPU test of triangular solves of many large factors against a few right-hand
sides at the limit of the one-launch form's shared memory: its rule has to
count the columns that the launch takes (1, 2, 4 or 8), or leave the solve to
the recursive form.

85 factors of order 3375 (leaves of 17^3 nodes): five columns, taken as eight,
need 225 792 bytes.  Reference: each column's own solve (1e-11, both are
backward-stable solves with the same factors)."""

import numpy as np
import pytest

import workloads as W
from oracle import adaptive as ad

pytestmark = pytest.mark.gpu
torch = pytest.importorskip("torch")


@pytest.mark.parametrize("nrhs", [5])
def test_columns_rounded_up_in_the_size_rule(nrhs):
    if not torch.cuda.is_available():
        pytest.skip("no CUDA device")
    import paper_2503_17535_gb300 as P
    p = 17
    pr = W.elliptic_3d()
    leaves = [(2, (i, j, k)) for i in range(4) for j in range(4) for k in range(4)]
    for corner in ((0, 0, 0), (3, 0, 0), (0, 3, 3)):
        leaves.remove((2, corner))
        leaves += ad.children_of(2, corner)
    t = P.adaptive_tree(ad.sort_leaves(leaves), pr.lo, pr.hi)
    x, _ = P.hps_nodes(t, p, p - 2)
    nl, ppl, nr = P.hps_sizes(t, p, p - 2)
    assert nl == 85
    cf = pr.coeffs(x)
    d = lambda v: torch.from_numpy(np.ascontiguousarray(v)).cuda()  # noqa: E731
    h = P.hps_build(t, p, p - 2, P.HPS_DTN, a=d(cf["a"].reshape(nl, ppl)), b=[d(v.reshape(nl, ppl)) for v in cf["b"]],
                    c=d(cf["c"].reshape(nl, ppl)), lazy_root=True)
    gen = torch.Generator(device="cuda").manual_seed(7)
    z = lambda *s: torch.randn(*s, dtype=torch.float64, device="cuda", generator=gen)  # noqa: E731
    g, f, u = z(nrhs, nr), z(nrhs, nl, ppl), z(nrhs, nl, ppl)
    P.hps_solve_batched(h, nrhs, g, u, f=f)
    one = torch.empty((nl, ppl), dtype=torch.float64, device="cuda")
    for k in range(nrhs):
        P.hps_solve(h, g[k].contiguous(), one, f=f[k].contiguous())
        assert float((one - u[k]).abs().max()) <= 1e-11 * float(one.abs().max())
