"""GPU tests of adaptive solves whose number of right-hand sides changes from
call to call on one operator: the workspace's task tables hold the strides of one
number, and are written while the solve before may still read the old ones.

Reference: the first solve of a second operator (the same kernels on the same
data: equal up to the order of columns in a launch, 1e-12)."""

import numpy as np
import pytest

import workloads as W
from oracle import adaptive as ad

pytestmark = pytest.mark.gpu
torch = pytest.importorskip("torch")


@pytest.fixture(scope="module")
def setup():
    if not torch.cuda.is_available():
        pytest.skip("no CUDA device")
    import paper_2503_17535_gb300 as P
    p, pr = 6, W.elliptic_3d()
    leaves = [(1, (i, j, k)) for i in range(2) for j in range(2) for k in range(2) if (i, j, k) != (0, 0, 0)]
    t = P.adaptive_tree(ad.sort_leaves(leaves + ad.children_of(1, (0, 0, 0))), pr.lo, pr.hi)
    x, _ = P.hps_nodes(t, p, p - 2)
    nl, ppl, nr = P.hps_sizes(t, p, p - 2)
    cf = pr.coeffs(x)
    d = lambda v: torch.from_numpy(np.ascontiguousarray(v)).cuda()  # noqa: E731
    a, b, c = d(cf["a"].reshape(nl, ppl)), [d(v.reshape(nl, ppl)) for v in cf["b"]], d(cf["c"].reshape(nl, ppl))
    rng = np.random.default_rng(3)
    g, f, f0 = d(rng.standard_normal((4, nr))), d(rng.standard_normal((4, nl, ppl))), d(rng.standard_normal((nl, ppl)))
    build = lambda lazy: P.hps_build(t, p, p - 2, P.HPS_DTN, a=a, b=b, c=c, f=f0, lazy_root=lazy)  # noqa: E731
    return P, build, g, f


def _solve(P, h, n, g, f):
    u = torch.full((n,) + f.shape[1:], float("nan"), dtype=torch.float64, device="cuda")
    P.hps_solve_batched(h, n, g[:n].contiguous(), u, f=f[:n].contiguous())
    v = torch.full_like(u, float("nan"))
    P.hps_solve_batched(h, n, g[:n].contiguous(), v)
    return torch.stack([u, v])


@pytest.mark.parametrize("lazy", [False, True], ids=["explicit", "lazy"])
def test_fewer_right_hand_sides_after_more(setup, lazy):
    P, build, g, f = setup
    h = build(lazy)
    for n in (3, 1, 2, 4, 3):
        got, ref = _solve(P, h, n, g, f), _solve(P, build(lazy), n, g, f)
        assert bool((got - ref).abs().max() <= 1e-12 * ref.abs().max())


def test_numbers_alternate_on_a_stream_of_its_own(setup):
    """No synchronisation between the calls, and work before them on the stream."""
    P, build, g, f = setup
    h = build(False)
    ref = {n: _solve(P, build(False), n, g, f)[0] for n in (1, 3, 4)}
    st = torch.cuda.Stream()
    busy = torch.randn(4096, 4096, device="cuda")
    ins = {n: (g[:n].contiguous(), f[:n].contiguous()) for n in ref}
    torch.cuda.synchronize()
    got = []
    with torch.cuda.stream(st):
        for n in (3, 1, 4, 1, 3, 4, 3, 1) * 3:
            for _ in range(4):
                busy = busy @ busy * 1e-3
            got.append((n, torch.empty((n,) + f.shape[1:], dtype=torch.float64, device="cuda")))
            P.hps_solve_batched(h, n, ins[n][0], got[-1][1], f=ins[n][1])
    torch.cuda.synchronize()
    for n, u in got:
        assert bool((u - ref[n]).abs().max() <= 1e-12 * ref[n].abs().max())


@pytest.mark.parametrize("k", [1, 4, 12, 30])
def test_a_workspace_that_could_not_grow_is_made_anew(setup, k):
    P, build, g, f = setup
    h = build(False)
    ref = _solve(P, h, 1, g, f)
    P.hps_debug_fail_alloc(k)
    try:
        with pytest.raises(P.HPSError):
            _solve(P, h, 3, g, f)
    finally:
        P.hps_debug_fail_alloc(0)
    assert torch.equal(_solve(P, h, 1, g, f), ref)
