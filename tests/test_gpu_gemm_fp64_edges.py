"""GPU tests of the FP64-pipe product at the edges of its tiles (32 x 8, 16 x 16
and 8 x 32, chosen by the padding) and of its 32-step stages of K.

Reference: the product in FP64 on the host; bound 4 (K + 8) 2^-53 times
|A| |B| (entries' |re| + |im| for complex data: the 3M sums) plus |C|, times the
factors alpha and beta -- the a priori bound of a K-term sum and its epilogue,
doubled for the reference's own rounding and again for the 3M sums."""

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


SHAPES = [(1, 9, 1, 1), (7, 31, 3, 5), (8, 33, 4, 2), (9, 17, 31, 3), (16, 16, 32, 1), (17, 15, 33, 70), (24, 40, 64, 2),
          (31, 9, 65, 1), (33, 64, 100, 4), (40, 1000, 5, 1), (300, 10, 36, 2), (129, 130, 67, 1), (3, 12, 2, 66000)]


@pytest.mark.parametrize("m,n,k,batch", SHAPES, ids=["x".join(map(str, s)) for s in SHAPES])
@pytest.mark.parametrize("alpha,beta", [(-1.0, 1.0), (1.0, 0.0), (0.75, -1.25), (2.0, 0.0)])
@pytest.mark.parametrize("cplx", [False, True], ids=["real", "complex"])
def test_tiles_and_stages(P, m, n, k, batch, alpha, beta, cplx):
    rng = np.random.default_rng(m + 3 * n + 7 * k)
    z = (lambda *s: rng.standard_normal(s) + 1j * rng.standard_normal(s)) if cplx else lambda *s: rng.standard_normal(s)
    A, B, C0 = z(batch, k, m), z(batch, n, k), z(batch, n, m)   # each item's columns contiguous
    d = lambda v: torch.from_numpy(v.copy()).cuda()  # noqa: E731
    C = d(C0 if beta else C0 * np.nan)   # beta = 0 never reads C
    P.hps_gemm(d(A), d(B), C, alpha=alpha, beta=beta, mode=1)
    a1 = lambda v: np.abs(v.real) + np.abs(v.imag)  # noqa: E731
    ref = alpha * (B @ A) + (beta * C0 if beta else 0.0)
    bound = 4 * (k + 8) * 2.0 ** -53 * (abs(alpha) * (a1(B) @ a1(A)) + abs(beta) * a1(C0))
    assert np.all(np.abs(C.cpu().numpy() - ref) <= bound)
