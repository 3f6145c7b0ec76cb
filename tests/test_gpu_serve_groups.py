"""GPU test of the request server's grouping: requests with and without a new
source waiting on the same slots, more than one batch of each per slot, so that
a scheduling pass dispatches a slot's own batch between the slots it collects
for a group.  Every request is answered and equals its plain solve (1e-12: the
grouped products sum in another order)."""

import numpy as np
import pytest

import workloads as W
from test_gpu_parity import P, rel, sample_inputs  # noqa: F401

pytestmark = pytest.mark.gpu
torch = pytest.importorskip("torch")


@pytest.mark.parametrize("seed", range(8))
def test_mixed_heads_share_groups(P, seed):  # noqa: F811
    ops = [(W.e1_dtn_2d(), 8, 2), (W.e2_iti_2d(), 8, 2), (W.poisson_poly_2d(seed=0), 10, 1), (W.elliptic_3d(seed=2), 6, 1)]
    data, plain = [], []
    for pr, p, L in ops:
        t, x, a, b, c, f, g = sample_inputs(P, pr, p, L)
        cc = np.ascontiguousarray
        a, b, c, f, g = cc(a), [cc(v) for v in b], cc(c), cc(f), cc(g)
        kind = P.HPS_ITI if pr.kind == "iti" else P.HPS_DTN
        data.append((pr, p, t, kind, a, b, c, f, g))
        plain.append(P.hps_build(t, p, p - 2, kind, a=a, b=b, c=c, f=f, eta=pr.eta or 0.0))
    rng = np.random.default_rng(seed)
    reqs = []
    with P.Server(n_slots=4, n_streams=3, max_batch=2) as S:
        for i, (pr, p, t, kind, a, b, c, f, g) in enumerate(data):
            S.submit_build(i, t, p, p - 2, kind, a=a, b=b, c=c, f=f, eta=pr.eta or 0.0)
        for _ in range(60):
            i = int(rng.integers(0, 4))
            f, g = data[i][7], data[i][8]
            gn = (rng.standard_normal(g.shape) + (1j * rng.standard_normal(g.shape) if np.iscomplexobj(g) else 0)).astype(g.dtype)
            fn = 2.0 * f if rng.random() < 0.4 else None
            u = np.zeros_like(f)
            reqs.append((S.submit_solve(i, gn, u, f=fn), i, gn, fn, u))
        infos = [S.wait(t, check=False) for t, *_ in reqs]
    assert all(v["status"] == 0 for v in infos), [v for v in infos if v["status"]]
    for _, i, gn, fn, u in reqs:
        ref = np.zeros_like(u)
        P.hps_solve(plain[i], gn, ref, f=fn)
        assert rel(u, ref) <= 1e-12
    for h in plain:
        P.hps_free(h)
