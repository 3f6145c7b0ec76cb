"""GPU tests of the LU whose panels run beside the trailing updates: orders just
below and above the rule's limit, last panels of a few columns, one to four
matrices, and several threads at once on their own streams.

Reference: LAPACK's interchanges and the backward error bound
|L U - P A| <= 4 n 2^-53 |L| |U| + 2 n 2^-52 max|L| max|U| (the second term: the
digit products' rounding, relative to the largest entries of a row and a
column, in mode 0)."""

import threading

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


def _batch(n, batch, cplx, seed):
    rng = np.random.default_rng(seed)
    A = rng.standard_normal((batch, n, n))
    return A + 1j * rng.standard_normal((batch, n, n)) if cplx else A


def _factor(P, A, mode, stream=None):
    Ad = torch.from_numpy(np.ascontiguousarray(np.swapaxes(A, 1, 2))).cuda()
    torch.cuda.synchronize()
    _, ipiv, info = P.hps_getrf(Ad, mode=mode, stream=stream)
    assert int(info.abs().sum()) == 0
    return np.swapaxes(Ad.cpu().numpy(), 1, 2), ipiv.cpu().numpy()


@pytest.mark.parametrize("n,batch,cplx", [(270, 1, False), (310, 1, False), (545, 2, False), (1025, 1, False), (600, 4, False),
                                          (380, 1, True), (530, 1, True), (449, 3, True), (1000, 1, True)])
@pytest.mark.parametrize("mode", [0, 1], ids=["digits", "fp64"])
def test_matches_lapack(P, n, batch, cplx, mode):
    A = _batch(n, batch, cplx, n)
    F, ip = _factor(P, A, mode)
    for b in range(batch):
        assert np.array_equal(ip[b], sla.lu_factor(A[b])[1])
        L, U = np.tril(F[b], -1) + np.eye(n), np.triu(F[b])
        PA = A[b].copy()
        for j, p in enumerate(ip[b]):
            PA[[j, p]] = PA[[p, j]]
        extra = 2 * n * 2.0 ** -52 * np.abs(L).max() * np.abs(U).max()
        assert np.all(np.abs(L @ U - PA) <= 4 * n * 2.0 ** -53 * (np.abs(L) @ np.abs(U)) + extra)


def test_threads_on_their_own_streams(P):
    """More threads than the library keeps idle side streams, each with its own
    matrices: the factors of the same matrix are the same bits."""
    mats = [_batch(500 + 16 * (i % 4), 1, i % 2 == 1, i % 4) for i in range(12)]
    ref = [_factor(P, m, 0) for m in mats[:4]]
    out, errs = [None] * len(mats), []

    def work(i):
        try:
            s = torch.cuda.Stream()
            for _ in range(3):
                out[i] = _factor(P, mats[i], 0, stream=s.cuda_stream)
        except Exception as e:  # noqa: BLE001
            errs.append(e)

    ts = [threading.Thread(target=work, args=(i,)) for i in range(len(mats))]
    [t.start() for t in ts]
    [t.join() for t in ts]
    assert not errs, errs
    for i in range(len(mats)):
        assert np.array_equal(out[i][0], ref[i % 4][0]) and np.array_equal(out[i][1], ref[i % 4][1])
    P.hps_trim()
    assert np.array_equal(_factor(P, mats[0], 0)[0], ref[0][0])
