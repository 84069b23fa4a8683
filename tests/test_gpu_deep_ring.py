"""Networks whose edges span many levels (a deep ring of routed counts) at
n R >= 2^18, where the planner chooses between the persistent and the per-step
kernels (GPU): every entry of both forms and of the planner's choice equal, and
sampled replications equal the oracle's.
"""
import numpy as np
import pytest

from paper_2402_13259_gb300 import workloads as W

pytestmark = pytest.mark.gpu


@pytest.fixture(scope="module")
def Bd():
    import torch
    if not torch.cuda.is_available():
        pytest.fail("these tests need a CUDA GPU")
    from paper_2402_13259_gb300 import binding
    return binding


def _net(n, edges):
    row_ptr, col, prob = W.csr_from_edges(n, edges)
    w = np.zeros(n)
    w[::4] = 6.0
    arr = W.Arrivals(kind=W.ARR_SINUSOID, w=w, a=1.0, b=0.4, period=2.0, phase=0.1)
    return W.Network(n, row_ptr, col, prob, np.where(np.arange(n) % 2 == 0, 2, 9), np.linspace(0.8, 1.7, n), arr,
                     N0=(3 + np.arange(n) % 5).astype(np.int32))


def _complete(n):
    return _net(n, [(i, j, 0.9 / (n - 1 - i)) for i in range(n) for j in range(i + 1, n)])


def _two_wide(levels):
    e = [(2 * l + a, 2 * l + 2 + b, 0.4) for l in range(levels - 1) for a in range(2) for b in range(2)]
    return _net(2 * levels, e + [(0, 2 * levels - 1, 0.1)])


@pytest.mark.parametrize("scheme", [0, 1])
@pytest.mark.parametrize("make,size,R", [(_complete, 40, 6600), (_two_wide, 100, 1400)])
def test_deep_ring(Bd, orc, make, size, R, scheme):
    net = make(size)
    assert net.n * R >= 1 << 18
    h = Bd.EulerNet(net)
    got = {}
    try:
        for form in (-1, 1, 2):
            h.set_option(Bd.OPT_FORM, form)
            got[form] = h.simulate(scheme, 0.1, 1.5, R, 17, rep_begin=3).cpu().numpy()
    finally:
        h.close()
    assert np.array_equal(got[1], got[2]) and np.array_equal(got[-1], got[2])
    rp = Bd.split_stats(got[1], net.n, R)["rep"]
    for r in (0, R // 2, R - 1):
        want = orc.simulate(net, scheme, 0.1, 1.5, 1, 17, rep_begin=3 + r)["rep"][0]
        assert np.array_equal(rp[r], want), r


def _chain(n):
    return _net(n, [(i, i + 1, 0.6) for i in range(n - 1)])


@pytest.mark.parametrize("make,size,R", [(_two_wide, 100, 1400), (_chain, 4000, 1)])
def test_captured_call(Bd, make, size, R):
    """A call whose eager form is per-step kernels, captured by the caller and
    replayed."""
    import torch
    net = make(size)
    h = Bd.EulerNet(net)
    try:
        assert h.plan(1, R)["form"] == 2
        want = h.simulate(1, 0.1, 1.0, R, 5).cpu().numpy()
        stats = torch.empty(Bd.stats_len(net.n, R), dtype=torch.int64, device="cuda")
        g = torch.cuda.CUDAGraph()
        with torch.cuda.graph(g):
            h.simulate(1, 0.1, 1.0, R, 5, stats=stats, check=False)
        for _ in range(2):
            stats.fill_(-1)
            g.replay()
            h.status()
            assert np.array_equal(stats.cpu().numpy(), want)
    finally:
        h.close()
