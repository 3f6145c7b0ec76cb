"""GPU tests of the substitutions with one to eight threads per column, at the
edges of their rules: panels narrower than the kernel's row count with
interchanges that land just below them, last panels and diagonal blocks of a
few rows, column counts that leave warps without columns, batches from one
matrix to thousands (each of the four splits).

References: for the factorisation LAPACK's interchanges and the backward error
bound |L U - P A| <= 4 n 2^-53 |L| |U|; for the solves the one-column solve
with the same factors (1e-11: both are backward-stable)."""

import numpy as np
import pytest
import scipy.linalg as sla

import workloads as W

pytestmark = pytest.mark.gpu
torch = pytest.importorskip("torch")


@pytest.fixture(scope="module")
def P():
    if not torch.cuda.is_available():
        pytest.skip("no CUDA device")
    import paper_2503_17535_gb300 as P
    return P


@pytest.mark.parametrize("n,batch,width", [(70, 1, 8), (150, 2, 16), (201, 3, 24), (333, 1, 32), (47, 4000, 32), (77, 700, 32),
                                           (260, 90, 32), (190, 9, 32)])
@pytest.mark.parametrize("cplx", [False, True], ids=["real", "complex"])
def test_interchanges_near_and_far(P, n, batch, width, cplx):
    rng = np.random.default_rng(n + batch)
    A = 0.1 * rng.standard_normal((batch, n, n))
    if cplx:
        A = A + 0.1j * rng.standard_normal((batch, n, n))
    # dominant entries a few rows off the diagonal: pivots just below the panel
    for b in range(min(batch, 64)):
        perm = np.argsort(np.arange(n) + rng.uniform(0, 12, n))
        A[b, perm, np.arange(n)] += 3.0
    Ad = torch.from_numpy(np.ascontiguousarray(np.swapaxes(A, 1, 2))).cuda()
    old = P.hps_tune_get("lu_panel_nb_few")
    P.hps_tune_set("lu_panel_nb_few", width)
    try:
        _, ipiv, info = P.hps_getrf(Ad, mode=1)
    finally:
        P.hps_tune_set("lu_panel_nb_few", old)
    assert int(info.abs().sum()) == 0
    F, ip = np.swapaxes(Ad.cpu().numpy(), 1, 2), ipiv.cpu().numpy()
    for b in sorted({0, min(63, batch - 1), batch - 1}):
        assert np.array_equal(ip[b], sla.lu_factor(A[b])[1])
        L, U = np.tril(F[b], -1) + np.eye(n), np.triu(F[b])
        PA = A[b].copy()
        for j, p in enumerate(ip[b]):
            PA[[j, p]] = PA[[p, j]]
        assert np.all(np.abs(L @ U - PA) <= 4 * n * 2.0 ** -53 * (np.abs(L) @ np.abs(U)))


@pytest.mark.parametrize("kind,p,L,nrhs", [("dtn2", 10, 0, 17), ("dtn2", 9, 3, 33), ("dtn2", 10, 4, 130), ("dtn2", 8, 5, 65),
                                           ("dtn3", 7, 2, 40), ("iti", 10, 1, 17), ("iti", 9, 3, 40), ("iti", 8, 4, 33)])
def test_many_columns_match_one(P, kind, p, L, nrhs):
    pr = {"dtn2": W.elliptic_2d, "dtn3": W.elliptic_3d}.get(kind, lambda: W.helmholtz_bumps_2d(seed=1, k=6.0))()
    t = P.uniform_tree(pr.dim, L, pr.lo, pr.hi)
    x, _ = P.hps_nodes(t, p, p - 2)
    nl, ppl, nr = P.hps_sizes(t, p, p - 2)
    cf = pr.coeffs(x)
    g = torch.Generator(device="cuda").manual_seed(p)
    dt = torch.complex128 if kind == "iti" else torch.float64
    d = lambda v: torch.from_numpy(np.ascontiguousarray(v).reshape(nl, ppl)).cuda()  # noqa: E731
    h = P.hps_build(t, p, p - 2, P.HPS_ITI if kind == "iti" else P.HPS_DTN, a=d(cf["a"]), b=[d(v) for v in cf["b"]],
                    c=d(cf["c"]), eta=pr.eta or 0.0)
    f = torch.randn((nrhs, nl, ppl), dtype=dt, device="cuda", generator=g)
    gb = torch.randn((nrhs, nr), dtype=dt, device="cuda", generator=g)
    u, one = torch.empty_like(f), torch.empty((1, nl, ppl), dtype=dt, device="cuda")
    P.hps_solve_batched(h, nrhs, gb, u, f=f)
    for k in (0, nrhs // 2, nrhs - 1):
        P.hps_solve(h, gb[k], one, f=f[k])
        assert float((one[0] - u[k]).abs().max()) <= 1e-11 * float(one.abs().max())
