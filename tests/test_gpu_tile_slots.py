"""The persistent form's slot kernel against the oracle (GPU) at the sizes
where its index arithmetic has edges: one replication to a tile, tiles that do
not divide the replications, a unit count just below, at and above a whole
number of warps, units listed and drawn in place, routed counts kept for more
than two slots, no external arrivals, and several launches of tiles.  Whole
numbers: every entry must be equal.
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


def _net(n, skip, arrivals=True, heavy=True):
    """A chain 0 -> 1 -> ... -> n-1 with edges i -> i + skip beside it (ring
    depth skip + 1); few servers, so that many units have x > m."""
    edges = []
    for i in range(n - 1):
        edges.append((i, i + 1, 0.6))
        if skip > 1 and i + skip < n:
            edges.append((i, i + skip, 0.3))
    row_ptr, col, prob = W.csr_from_edges(n, edges)
    w = np.zeros(n)
    if arrivals:
        w[::3] = 12.0
    arr = W.Arrivals(kind=W.ARR_SINUSOID, w=w, a=1.0, b=0.5, period=3.0, phase=0.1)
    m = np.where(np.arange(n) % 2 == 0, 2, 9) if heavy else np.full(n, 500)
    return W.Network(n, row_ptr, col, prob, m, np.linspace(0.8, 1.7, n), arr,
                     N0=(7 + np.arange(n) % 5).astype(np.int32))


@pytest.mark.parametrize("scheme", [0, 1])
@pytest.mark.parametrize("n,skip,R,tile,block", [
    (1, 1, 1, 1, 32),        # one unit
    (3, 1, 153, 0, 0),       # the planner's tiles, one more replication than SMs
    (5, 4, 77, 8, 32),       # ring depth 5, listed, a ragged last tile
    (31, 2, 33, 32, 64),     # 992 units a tile: 31 warps' worth, listed
    (33, 3, 64, 32, 512),    # 1,056 units: 33 warps' worth
    (17, 2, 250, 64, 64),    # 1,088 units, last tile 58 replications
    (40, 2, 400, 0, 0),      # the planner's tiles
])
def test_slots_equal_oracle(Bd, orc, scheme, n, skip, R, tile, block):
    for arrivals, heavy in ((True, True), (True, False), (False, True)):
        net = _net(n, skip, arrivals, heavy)
        h = Bd.EulerNet(net)
        try:
            h.set_option(Bd.OPT_FORM, 1)
            if tile:
                h.set_option(Bd.OPT_TILE_REPS, tile)
                h.set_option(Bd.OPT_BLOCK, block)
            got = h.simulate(scheme, 0.1, 1.7, R, 11, rep_begin=5).cpu().numpy()
        finally:
            h.close()
        want = orc.simulate(net, scheme, 0.1, 1.7, R, 11, rep_begin=5)["stats"]
        bad = np.nonzero(got != want)[0]
        assert bad.size == 0, f"{bad.size} entries differ, first {bad[:5].tolist()}"


@pytest.mark.parametrize("scheme", [0, 1])
def test_small_large_small_on_one_handle(Bd, orc, scheme):
    """Calls of different size on one handle share its scratch."""
    net = _net(12, 2)
    h = Bd.EulerNet(net)
    try:
        for R in (3, 2000, 3, 500):
            got = h.simulate(scheme, 0.1, 0.9, R, 21).cpu().numpy()
            want = orc.simulate(net, scheme, 0.1, 0.9, R, 21)["stats"]
            assert np.array_equal(got, want), R
    finally:
        h.close()


@pytest.mark.parametrize("scheme", [0, 1])
@pytest.mark.parametrize("fan", [1, 3, 4, 9])
def test_fan_in(Bd, orc, scheme, fan):
    """A station with more in-edges than its record holds (three)."""
    row_ptr, col, prob = W.csr_from_edges(fan + 1, [(i, fan, 0.9) for i in range(fan)])
    arr = W.Arrivals(kind=W.ARR_SINUSOID, w=np.full(fan + 1, 9.0), a=1.0, b=0.2, period=5.0)
    net = W.Network(fan + 1, row_ptr, col, prob, np.full(fan + 1, 4), np.full(fan + 1, 1.3), arr)
    h = Bd.EulerNet(net)
    try:
        h.set_option(Bd.OPT_FORM, 1)
        got = h.simulate(scheme, 0.1, 2.0, 40, 3).cpu().numpy()
    finally:
        h.close()
    assert np.array_equal(got, orc.simulate(net, scheme, 0.1, 2.0, 40, 3)["stats"])


def test_batch_of_both_schemes(Bd, orc):
    """Both schemes in one batch run side by side, small tiles in place and
    larger ones listed, and the batch runs again on the same plan."""
    nets = [_net(n, 2, True, n % 2 == 0) for n in (1, 4, 9, 40, 41, 120)]
    runs = [(j % 2, 0.1, 1.0 + 0.3 * j, R, 50 + j) for j, R in enumerate((7, 200, 33, 90, 64, 130))]
    hs = [Bd.EulerNet(x) for x in nets]
    b = Bd.Batch(hs, runs)
    try:
        for _ in range(2):
            got = [s.cpu().numpy() for s in b.run()]
            for net, r, g in zip(nets, runs, got):
                assert np.array_equal(g, orc.simulate(net, r[0], r[1], r[2], r[3], r[4])["stats"]), r
    finally:
        b.close()
        for h in hs:
            h.close()
