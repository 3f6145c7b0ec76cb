"""GPU tests of the last bits of the tensor-core FP64 product: the resolution of
its fixed-point sum at short inner dimensions and the rounding of entries far
below their row's largest.

With n products summed per output (2K for a component of a complex product),
scaled so that every factor is below 1, the sum is below n and keeps
lsb = min(62, 63 - ceil(log2 n)) fraction bits up to 128 of them."""

import math
from fractions import Fraction

import numpy as np
import pytest

pytestmark = pytest.mark.gpu
torch = pytest.importorskip("torch")


@pytest.fixture(scope="module")
def P():
    if not torch.cuda.is_available():
        pytest.skip("no CUDA device")
    import paper_2503_17535_gb300 as P
    return P


def _product(P, A, B, alpha, beta=0.0):
    """alpha A B, entry (0, 0); A (1, m, k), B (1, k, n)."""
    dev = lambda x: torch.from_numpy(np.ascontiguousarray(np.swapaxes(x, 1, 2))).cuda()  # noqa: E731
    C = torch.zeros((1, B.shape[2], A.shape[1]), dtype=torch.from_numpy(A).dtype, device="cuda")
    P.hps_gemm(dev(A), dev(B), C, alpha=alpha, beta=beta)
    return C


@pytest.mark.parametrize("alpha,beta", [(1.0, 0.0), (-1.0, 1.0), (0.5, 0.0)], ids=["set", "subtract", "general"])
@pytest.mark.parametrize("cplx", [False, True], ids=["real", "complex"])
@pytest.mark.parametrize("k", [4, 8, 16, 17, 32, 64])
def test_a_sum_of_one_unit_survives(P, k, cplx, alpha, beta):
    """A row (0.5, 0, 2^-30, 0 ..) times a column (0, 0.5, 2^(30 - lsb), 0 ..):
    the product is one unit of the fixed point, exactly representable, and both
    small factors are one digit each, so that nothing is dropped or rounded.
    One bit less loses it (ties to even)."""
    n = (2 if cplx else 1) * k
    lsb = min(62, 63 - math.ceil(math.log2(n)))
    dt = np.complex128 if cplx else np.float64
    A, B = np.zeros((1, 40, k), dt), np.zeros((1, k, 40), dt)
    A[0, :, 0], A[0, :, 2] = 0.5, 2.0 ** -30
    B[0, 1, :], B[0, 2, :] = 0.5, 2.0 ** (30 - lsb)
    C = _product(P, A, B, alpha, beta)
    assert bool((C == alpha * 2.0 ** -lsb).all())


@pytest.mark.parametrize("sign", [1.0, -1.0])
@pytest.mark.parametrize("below", [11, 30, 42, 43, 44, 50, 53, 60])
@pytest.mark.parametrize("part", [0.25, 0.9375])
def test_small_entries_round_to_nearest(P, below, part, sign):
    """63 entries (m + part) 2^-62, m even, 2^below below the row's largest, times
    63 / 64 each (one digit, nothing dropped).  Every entry rounds to the nearest
    multiple of 2^-62: the sum is off by at most 63 min(part, 1 - part) 2^-62 plus
    half a unit of 2^-57; rounded the other way, by 63 max(part, 1 - part) 2^-62,
    more than twice that for part = 0.9375."""
    m = 2 ** (62 - below - 1) if below < 61 else 2
    t = float(sign * (Fraction(m) + Fraction(part)) / 2 ** 62)
    exact1 = Fraction(t)
    A, B = np.full((1, 40, 64), t), np.full((1, 64, 40), 63.0 / 64)
    A[0, :, 0], B[0, 0, :] = 0.5, 0.0
    C = _product(P, A, B, 1.0)
    exact = 63 * exact1 * Fraction(63, 64)
    bits = float(abs(exact1 * 2 ** 62 - round(exact1 * 2 ** 62)))   # what FP64 could hold of the part
    lim = 63 * bits * 2.0 ** -62 + 2.0 ** -58 + 2.0 ** -53 * abs(float(exact))
    err = [abs(float(Fraction(float(v)) - exact)) for v in torch.unique(C).cpu()]
    assert max(err) <= lim, (max(err) / 2.0 ** -58, lim / 2.0 ** -58)
