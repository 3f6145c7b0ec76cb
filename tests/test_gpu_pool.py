"""GPU test of the device memory kept after frees: bounded by a sixteenth of
the device's memory, counted as free when the next build is planned, given
back by hps_trim and, when the device runs short, to other allocations of the
process."""

import numpy as np
import pytest

import workloads as W
from test_gpu_parity import P, dev, rel, sample_inputs  # noqa: F401

pytestmark = pytest.mark.gpu
torch = pytest.importorskip("torch")


def test_kept_memory_is_bounded_and_given_back(P):  # noqa: F811
    pr = W.helmholtz_bumps_2d(seed=1)
    p, L = 16, 5
    inputs = sample_inputs(P, pr, p, L)
    t, x, a, b, c, f, g = inputs
    args = dict(a=dev(a), b=[dev(v) for v in b], c=dev(c), f=dev(f), eta=pr.eta)
    u = [torch.empty(f.shape, dtype=torch.complex128, device="cuda") for _ in range(2)]
    gd = dev(g)
    torch.cuda.synchronize()
    P.hps_trim()
    free0, total = torch.cuda.mem_get_info()
    for k in range(2):
        h = P.hps_build(t, p, p - 2, P.HPS_ITI, **args)
        P.hps_solve(h, gd, u[k])
        P.hps_free(h)
        torch.cuda.synchronize()
        kept = free0 - torch.cuda.mem_get_info()[0]
        assert 0 <= kept <= total // 16 + (64 << 20)
    assert kept > 1 << 30                       # the operator's buffers wait for the next build
    P.hps_trim()
    assert free0 - torch.cuda.mem_get_info()[0] <= 64 << 20
    assert np.array_equal(u[0].cpu().numpy(), u[1].cpu().numpy())
