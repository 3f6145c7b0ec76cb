"""GPU tests of the tensor-core FP64 product at the edges of its tiles (128 x 64
and 128 x 32, either orientation), of its accumulation chunks (64 and 128
summed products) and of its exact digit sums.

Reference: the exact rational value of sampled dot products.  Bound, with
K' summed products per output (2K for a component of a complex product),
e and f the exponents of the row's and column's largest magnitude:

  |C - exact| <= (K' 2^-58.9 + chunks 2^-lsb) 2^(e + f) + 2^-52 (|exact| + |C0|)

operand rounding K' 2^-62, dropped digit pairs 7 K' 2^-62 (both below
K' 2^-58.9), half a unit of 2^-lsb per chunk with lsb = 57 up to 64 summed
products (rounded up to a multiple of 16 per real product), 56 up to 128 and
63 - ceil(log2 K') in chunks of 128 beyond, and the roundings to FP64.
"""

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


def _colmajor(x):
    return torch.from_numpy(np.ascontiguousarray(np.swapaxes(x, 1, 2))).cuda()


def _product(P, A, B, C0):
    C = _colmajor(C0)
    P.hps_gemm(_colmajor(A), _colmajor(B), C, alpha=-1.0, beta=1.0)
    return np.swapaxes(C.cpu().numpy(), 1, 2)


def _exp(x):
    return math.frexp(float(np.abs(x).max()))[1] if np.any(x) else 0


def _check(a, b, c0, got):
    """One real output: a, b the summed factors, got = c0 - a . b."""
    exact = Fraction(float(c0)) - sum(Fraction(float(x)) * Fraction(float(y)) for x, y in zip(a, b))
    return exact, abs(Fraction(float(got)) - exact)


def _limit(kp, scale, exact, c0):
    lsb = 57 if kp <= 64 else 56 if kp <= 128 else 63 - math.ceil(math.log2(kp))
    chunks = -(-kp // 128)
    return (kp * 2.0 ** -58.9 + chunks * 2.0 ** -lsb) * scale + 2.0 ** -52 * (abs(float(exact)) + abs(float(c0)))


SHAPES = [(127, 31, 64, 1), (128, 32, 65, 2), (129, 33, 128, 1), (130, 63, 129, 1), (64, 64, 144, 2), (33, 65, 16, 3),
          (31, 257, 48, 200), (36, 129, 17, 400), (257, 96, 33, 2), (192, 128, 260, 1)]


@pytest.mark.parametrize("m,n,k,batch", SHAPES, ids=["x".join(map(str, s)) for s in SHAPES])
@pytest.mark.parametrize("cplx", [False, True], ids=["real", "complex"])
def test_tile_and_chunk_edges(P, m, n, k, batch, cplx):
    rng = np.random.default_rng(m + 3 * n + 7 * k)
    z = (lambda s: rng.standard_normal(s) + 1j * rng.standard_normal(s)) if cplx else rng.standard_normal
    A, B, C0 = z((batch, m, k)), z((batch, k, n)), z((batch, m, n))
    A *= np.ldexp(1.0, rng.integers(-30, 31, (batch, m, 1)))
    C = _product(P, A, B, C0)
    picks = [(0, 0, 0), (batch - 1, m - 1, n - 1), (batch - 1, 0, n - 1), (0, m - 1, 0)]
    picks += [(int(rng.integers(batch)), int(rng.integers(m)), int(rng.integers(n))) for _ in range(20)]
    kp = -(-k // 16) * 16 * (2 if cplx else 1)
    for b, i, j in picks:
        a, x = A[b, i], B[b, :, j]
        if not cplx:
            ex, err = _check(a, x, C0[b, i, j], C[b, i, j])
            assert float(err) <= _limit(kp, 2.0 ** (_exp(a) + _exp(x)), ex, C0[b, i, j])
            continue
        scale = 2.0 ** (max(_exp(a.real), _exp(a.imag)) + max(_exp(x.real), _exp(x.imag)))
        for left, right, c0, got in ((np.r_[a.real, a.imag], np.r_[x.real, -x.imag], C0[b, i, j].real, C[b, i, j].real),
                                     (np.r_[a.real, a.imag], np.r_[x.imag, x.real], C0[b, i, j].imag, C[b, i, j].imag)):
            ex, err = _check(left, right, c0, got)
            assert float(err) <= _limit(kp, scale, ex, c0)
    # every entry, against FP64
    ref = C0 - np.matmul(A, B)
    mag = np.matmul(np.abs(A), np.abs(B)) + np.abs(C0)
    amax = np.abs(A).max(axis=2)[:, :, None] * np.abs(B).max(axis=1)[:, None, :]
    assert np.all(np.abs(C - ref) <= (2 * k + 8) * 2.0 ** -52 * mag + kp * 2.0 ** -54 * amax)


@pytest.mark.parametrize("k", [64, 128, 256])
@pytest.mark.parametrize("sign", [1.0, -1.0])
def test_largest_digit_sums_stay_exact(P, k, sign):
    """Every entry's digits are the leading 64 and six times -128 (then 0), so
    that every diagonal's sum reaches its bound; the product is one rational
    number, and the digits represent the entries exactly."""
    v = (64 * 2 ** 56 - 128 * sum(2 ** (8 * j) for j in range(1, 7))) / 2.0 ** 62
    m, n = 130, 70
    A, B = np.full((1, m, k), v), np.full((1, k, n), sign * v)
    C0 = np.zeros((1, m, n))
    C = _product(P, A, B, C0)
    ex = -Fraction(v) * Fraction(sign * v) * k
    lim = _limit(k, 1.0, ex, 0.0)
    assert np.all(C == C[0, 0, 0]) and float(abs(Fraction(float(C[0, 0, 0])) - ex)) <= lim
