"""GPU tests of the triangular solves against few right-hand sides (one CTA or
one cluster per matrix, up to 16 columns) at the edges of their blocks: factors
of less than one 32-row block, ragged last blocks, clusters of 2 to 16 CTAs,
column counts on both sides of the kernels' groups (1, 2, 4, 8) and of their
limit (16, beyond which the recursive solves run).

References: the oracle's solution for the first and the last column (1e-10,
the repository's bar), the other columns against their own one-column solve
(1e-11: both are backward-stable solves with the same factors), and the adjoint
identity Re<ubar, u> = Re<gbar, g> + Re<fbar, f>."""

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


CASES = [("dtn2", 5, 2, False), ("dtn2", 13, 2, True), ("iti", 6, 1, False), ("iti", 13, 2, True), ("iti", 10, 3, False),
         ("dtn3", 5, 1, True), ("dtn3", 8, 1, False), ("dtn3", 7, 2, False)]


@pytest.mark.parametrize("kind,p,L,lazy", CASES, ids=["%s-p%d-L%d-%s" % (c[0], c[1], c[2], "lazy" if c[3] else "explicit")
                                                      for c in CASES])
@pytest.mark.parametrize("nrhs", [1, 2, 3, 5, 8, 9, 16, 17])
def test_new_sources_and_adjoint(P, kind, p, L, lazy, nrhs):
    pr = {"dtn2": W.elliptic_2d, "dtn3": W.elliptic_3d}.get(kind, lambda: W.helmholtz_bumps_2d(seed=1, k=6.0))()
    t = P.uniform_tree(pr.dim, L, pr.lo, pr.hi)
    x, xb = P.hps_nodes(t, p, p - 2)
    nl, ppl, nr = P.hps_sizes(t, p, p - 2)
    cf = pr.coeffs(x)
    rng = np.random.default_rng(p + L)
    cdt = np.complex128 if kind == "iti" else np.float64
    z = lambda *s: (rng.standard_normal(s) + (1j * rng.standard_normal(s) if kind == "iti" else 0)).astype(cdt)  # noqa: E731
    a, b, c = cf["a"].reshape(nl, ppl), [v.reshape(nl, ppl) for v in cf["b"]], cf["c"].reshape(nl, ppl)
    f, g, ub = z(nrhs, nl, ppl), z(nrhs, nr), z(nrhs, nl, ppl)
    d = lambda v: torch.from_numpy(np.ascontiguousarray(v)).cuda()  # noqa: E731
    h = P.hps_build(t, p, p - 2, P.HPS_ITI if kind == "iti" else P.HPS_DTN, a=d(a), b=[d(v) for v in b], c=d(c),
                    eta=pr.eta or 0.0, lazy_root=lazy)
    u = torch.empty((nrhs, nl, ppl), dtype=torch.from_numpy(f).dtype, device="cuda")
    P.hps_solve_batched(h, nrhs, d(g), u, f=d(f))
    one = torch.empty((1, nl, ppl), dtype=u.dtype, device="cuda")
    for k in range(nrhs):
        P.hps_solve(h, d(g[k]), one, f=d(f[k]))
        assert float((one[0] - u[k]).abs().max()) <= 1e-11 * float(one.abs().max())
    for k in {0, nrhs - 1}:
        s = O.build(pr.dim, pr.kind, p, p - 2, L, pr.lo, pr.hi, a, b, c, f[k], eta=pr.eta)
        uo = O.solve(s, g[k])
        assert np.abs(u[k].cpu().numpy() - uo).max() <= 1e-10 * np.abs(uo).max()
    gb, fb = torch.empty_like(d(g)), torch.empty_like(u)
    P.hps_solve_adjoint(h, d(ub), gb, fb, nrhs=nrhs)
    lhs = (np.conj(ub) * u.cpu().numpy()).real.sum(axis=(1, 2))
    rg, rf = (np.conj(gb.cpu().numpy()) * g).real.sum(axis=1), (np.conj(fb.cpu().numpy()) * f).real.sum(axis=(1, 2))
    scale = np.linalg.norm(ub.reshape(nrhs, -1), axis=1) * np.linalg.norm(u.cpu().numpy().reshape(nrhs, -1), axis=1)
    assert np.all(np.abs(lhs - rg - rf) <= 1e-10 * scale)
