"""GPU tests of the panel LU beyond the rows that fit its register form (8192):
taller panels go to the cluster's shared memory, the rest of the matrix to the
register panels, so that one factorisation runs both.

Reference: row by row |L U - P A| <= 4 n 2^-53 |L| |U| (the backward error bound of
Gaussian elimination, twice for complex products and twice for the reciprocal
multipliers), multipliers of at most 1 (|re| + |im| pivoting: sqrt 2), a permutation
that the interchanges give; the products are formed in FP64 on the GPU."""

import pytest

pytestmark = pytest.mark.gpu
torch = pytest.importorskip("torch")


@pytest.mark.parametrize("n", [8193, 8290])
@pytest.mark.parametrize("cplx", [False, True], ids=["real", "complex"])
def test_factors_of_a_tall_matrix(n, cplx):
    if not torch.cuda.is_available():
        pytest.skip("no CUDA device")
    import paper_2503_17535_gb300 as P
    dt = torch.complex128 if cplx else torch.float64
    gen = torch.Generator(device="cuda").manual_seed(n)
    A = torch.randn(n, n, dtype=dt, device="cuda", generator=gen)   # A.T in the library's column order
    A[0, ::3] = 2.0                                                 # ties in the first column
    F, ipiv, info = P.hps_getrf(A.clone()[None], mode=1)
    assert int(info.abs().sum()) == 0
    F = F[0].T
    perm = list(range(n))
    for j, p in enumerate(ipiv[0].tolist()):
        assert j <= p < n
        perm[j], perm[p] = perm[p], perm[j]
    L = torch.tril(F, -1)
    assert float(L.abs().max()) <= (2.0 ** 0.5 if cplx else 1.0) * (1 + 2.0 ** -40)
    L.diagonal().fill_(1.0)
    U = torch.triu(F)
    bound = 4 * n * 2.0 ** -53 * (L.abs() @ U.abs())
    err = (L @ U - A.T[torch.tensor(perm, device="cuda")]).abs()
    assert bool((err <= bound).all())
    # the first column's pivot: the largest magnitude, the lowest row on ties
    m = A[0].real.abs() + (A[0].imag.abs() if cplx else 0)
    assert int(ipiv[0, 0]) == int(torch.nonzero(m == m.max())[0])
