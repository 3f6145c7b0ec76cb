"""GPU test of downward passes whose complex maps are larger than L2 keeps, with
numbers of right-hand sides that are no multiple of four: those left over by
fours are taken in a launch of their own.

Reference: each right-hand side's own solve (1e-12 of its largest value: the
same sums, at most in another order of their partial sums)."""

import pytest

pytestmark = pytest.mark.gpu
torch = pytest.importorskip("torch")


@pytest.mark.parametrize("nrhs", [5, 7, 9, 14])
def test_columns_left_over(nrhs):
    if not torch.cuda.is_available():
        pytest.skip("no CUDA device")
    import paper_2503_17535_gb300 as P
    L, p = 6, 10    # every level: 64 (p - 2)^2 4^(L - 1) complex entries, 67 MB
    t = P.uniform_tree(2, L)
    nl, ppl, nr = P.hps_sizes(t, p, p - 2)
    gen = torch.Generator(device="cuda").manual_seed(nrhs)
    z = lambda *s: torch.randn(*s, dtype=torch.complex128, device="cuda", generator=gen)  # noqa: E731
    c = 400.0 * (1.0 - 0.3 * torch.rand(nl, ppl, dtype=torch.float64, device="cuda", generator=gen))
    h = P.hps_build(t, p, p - 2, P.HPS_ITI, c=c, f=z(nl, ppl), eta=20.0)
    g = z(nrhs, nr)
    u = torch.full((nrhs, nl, ppl), float("nan"), dtype=torch.complex128, device="cuda")
    P.hps_solve_batched(h, nrhs, g, u)
    one = torch.empty((nl, ppl), dtype=torch.complex128, device="cuda")
    for k in range(nrhs):
        P.hps_solve(h, g[k].contiguous(), one)
        assert float((one - u[k]).abs().max()) <= 1e-12 * float(one.abs().max())
