"""GPU test of the accuracy of new-source solves with ill-conditioned factors.

The dense impedance leaf matrix (boundary rows, then the operator's interior
rows) has diagonal blocks of its U factor with condition numbers of several
thousand.  64 such leaves are solved by a cluster each, with the precomputed
inverses of those blocks.  A substitution leaves a small residual L u - f
whatever the condition; a multiplication by an inverse does not.

Reference: the build's own solution for the same source, whose leaves are
solved by substitution.  Residual: max |L u - f| over the interior nodes of all
leaves, relative to max (|L| |u| + |f|).  Bar: four times the reference's, for the
rounding errors' chance, and two units."""

import numpy as np
import pytest

import workloads as W
from oracle import leaf as lf

pytestmark = pytest.mark.gpu
torch = pytest.importorskip("torch")


@pytest.mark.parametrize("p", [10, 12, 16])
@pytest.mark.parametrize("nrhs", [1, 3])
def test_residual_of_ill_conditioned_leaves(p, nrhs):
    if not torch.cuda.is_available():
        pytest.skip("no CUDA device")
    import paper_2503_17535_gb300 as P
    L = 3
    pr = W.helmholtz_bumps_2d(seed=1, k=20.0)
    t = P.uniform_tree(2, L, pr.lo, pr.hi)
    x, _ = P.hps_nodes(t, p, p - 2)
    nl, ppl, nr = P.hps_sizes(t, p, p - 2)
    cf = pr.coeffs(x)
    a, b, c = cf["a"].reshape(nl, ppl), [v.reshape(nl, ppl) for v in cf["b"]], cf["c"].reshape(nl, ppl)
    rng = np.random.default_rng(p)
    z = lambda *s: rng.standard_normal(s) + 1j * rng.standard_normal(s)  # noqa: E731
    f, g = z(nrhs, nl, ppl), np.zeros((nrhs, nr), complex)
    d = lambda v: torch.from_numpy(np.ascontiguousarray(v)).cuda()  # noqa: E731
    h = P.hps_build(t, p, p - 2, P.HPS_ITI, a=d(a), b=[d(v) for v in b], c=d(c), f=d(f[0]), eta=pr.eta, iti_leaf=1)
    u0 = torch.empty((nl, ppl), dtype=torch.complex128, device="cuda")
    u = torch.empty((nrhs, nl, ppl), dtype=torch.complex128, device="cuda")
    P.hps_solve(h, d(g[0]), u0)
    P.hps_solve_batched(h, nrhs, d(g), u, f=d(f))
    grid = np.indices((p, p)).reshape(2, -1)
    inner = np.nonzero(np.all((grid > 0) & (grid < p - 1), axis=0))[0]
    side = (pr.hi[0] - pr.lo[0]) / 2 ** L
    Ls = [lf.assemble_L(2, p, side, a[i], [v[i] for v in b], c[i])[inner] for i in range(nl)]

    def residual(u, f):
        r = max(float(np.abs(M.astype(np.clongdouble) @ u[i] - f[i][inner]).max()) for i, M in enumerate(Ls))
        return r / max(float((np.abs(M) @ np.abs(u[i]) + np.abs(f[i][inner])).max()) for i, M in enumerate(Ls))

    ref = residual(u0.cpu().numpy(), f[0])
    for k in range(nrhs):
        got = residual(u[k].cpu().numpy(), f[k])
        assert got <= 4 * ref + 2.0 ** -52, (got, ref)
