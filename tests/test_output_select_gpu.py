"""Nearest neighbours and threshold pairs at the edges of their kernels' steps
(256 threads, 8 loads each, 512 ranked candidates, rows kept in shared memory up
to 16,384 values), with many equal values too: both are selections, so they are
compared exactly."""
import numpy as np
import pytest

from paper_1911_04200_gb300 import jsim

pytestmark = pytest.mark.gpu


def matrix(n, kind, torch):
    g = torch.Generator(device="cuda")
    g.manual_seed(n)
    J = torch.rand(n, n, generator=g, device="cuda", dtype=torch.float64)
    if kind == "levels":
        J = torch.floor(J * 3) / 4  # three values: hundreds of ties at every cut
    elif kind == "zeros":
        J.zero_()
    elif kind == "close":
        J = 0.5 + J * 2.0 ** -40    # equal upper halves
    return J


@pytest.mark.parametrize("kind", ["random", "levels", "zeros", "close"])
@pytest.mark.parametrize("n,k", [(2, 1), (65, 64), (256, 64), (257, 10), (2049, 33), (4099, 1), (16385, 64)])
def test_topk_edges(gpu, n, k, kind):
    import torch
    J = matrix(n, kind, torch)
    with jsim.Context() as ctx:
        idx, val = ctx.topk(J, k)
    rows = torch.arange(n, device="cuda") if n <= 4099 else torch.tensor([0, 1, 8191, 16384], device="cuda")
    K = J[rows].clone()
    K[torch.arange(len(rows), device="cuda"), rows] = -1.0  # the sample itself last
    v, j = torch.sort(K, dim=1, descending=True, stable=True)  # ties keep the smaller index first
    assert torch.equal(idx.view(torch.int64)[rows], j[:, :k])
    assert torch.equal(val[rows], v[:, :k])


@pytest.mark.parametrize("below", [False, True])
@pytest.mark.parametrize("n,tau,cap", [(2, 0.5, 4), (257, 0.5, 1 << 20), (2049, 0.97, 1 << 20), (2050, 0.25, 5000),
                                       (2305, 0.0, 1 << 22), (2305, 2.0, 16)])
def test_threshold_edges(gpu, n, tau, cap, below):
    import torch
    J = matrix(n, "random", torch)
    keep = (J <= tau) if below else (J >= tau)
    i, j = torch.nonzero(torch.triu(keep, 1), as_tuple=True)
    with jsim.Context() as ctx:
        pi, pj, v, count = ctx.threshold(J, tau, below=below, cap=cap)
    assert count == len(i)
    w = min(count, cap)
    assert torch.equal(pi.view(torch.int64)[:w], i[:w]) and torch.equal(pj.view(torch.int64)[:w], j[:w])
    assert torch.equal(v[:w], J[i[:w], j[:w]])


@pytest.mark.parametrize("below", [False, True])
@pytest.mark.parametrize("tau", [0.0, -0.0, -0.25, 0.25, float("inf"), -float("inf"), 5e-324, -5e-324])
def test_threshold_orders_like_binary64(gpu, tau, below):
    # zeros of both signs, subnormals, infinities and NaNs pass as a binary64 compare has it
    import torch
    edge = [0.0, -0.0, 5e-324, -5e-324, 0.25, -0.25, float("inf"), -float("inf"), float("nan"), -float("nan"), 1.0, -1.0]
    n = 64
    J = torch.tensor(np.resize(np.array(edge), n * n).reshape(n, n)).cuda()
    keep = (J <= tau) if below else (J >= tau)
    i, j = torch.nonzero(torch.triu(keep, 1), as_tuple=True)
    with jsim.Context() as ctx:
        pi, pj, v, count = ctx.threshold(J, tau, below=below, cap=n * n)
    assert count == len(i)
    assert torch.equal(pi.view(torch.int64)[:count], i) and torch.equal(pj.view(torch.int64)[:count], j)
