"""GPU tests of the register-resident panel LU at the edges of its row split:
one, two or four threads per row (32, 64, 128 rows a CTA), chunks of clusters
that end inside a warp, last panels narrower than a segment, many matrices.

Reference: LAPACK's getrf -- identical interchanges, and factors within the
rounding of the factorisation: |L U - P A| <= 4 n 2^-53 |L| |U| entrywise (the
backward error bound n u / (1 - n u) |L| |U| of Gaussian elimination, times
two for the complex products and two for the reciprocal multipliers)."""

import numpy as np
import pytest
import scipy.linalg as sla

pytestmark = pytest.mark.gpu
torch = pytest.importorskip("torch")


@pytest.fixture(scope="module")
def P():
    if not torch.cuda.is_available():
        pytest.skip("no CUDA device")
    import paper_2503_17535_gb300 as P
    return P


CASES = [(1, 1), (5, 3), (16, 2), (31, 1), (32, 400), (33, 1), (63, 2), (65, 1), (97, 160), (127, 3), (129, 1), (257, 40),
         (513, 2), (530, 200), (1030, 1)]


@pytest.mark.parametrize("n,batch", CASES, ids=[f"{n}x{b}" for n, b in CASES])
@pytest.mark.parametrize("cplx", [False, True], ids=["real", "complex"])
def test_pivots_and_factors(P, n, batch, cplx):
    if n == 530 and cplx:
        batch = 20
    rng = np.random.default_rng(n + batch)
    A = rng.standard_normal((batch, n, n))
    if cplx:
        A = A + 1j * rng.standard_normal((batch, n, n))
    # exact ties in the first columns: the lowest current position wins
    A[:, ::3, 0] = 2.0
    A[:, 1::4, min(1, n - 1)] = -3.0
    Ad = torch.from_numpy(np.ascontiguousarray(np.swapaxes(A, 1, 2))).cuda()
    _, ipiv, info = P.hps_getrf(Ad, mode=1)
    assert int(info.abs().sum()) == 0
    F = np.swapaxes(Ad.cpu().numpy(), 1, 2)
    ip = ipiv.cpu().numpy()
    for b in sorted({0, batch // 2, batch - 1}):
        lu, piv = sla.lu_factor(A[b])
        assert np.array_equal(ip[b], piv)
        L, U = np.tril(F[b], -1) + np.eye(n), np.triu(F[b])
        PA = A[b].copy()
        for j, p in enumerate(ip[b]):
            PA[[j, p]] = PA[[p, j]]
        assert np.all(np.abs(L @ U - PA) <= 4 * n * 2.0 ** -53 * (np.abs(L) @ np.abs(U)))
