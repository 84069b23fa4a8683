"""Both forms at sizes where each runs in several pieces (GPU): the per-step
kernels over chunks of replications of their own choice, with rejection draws
over a whole horizon, and the persistent form over several launches of tiles.
The form is forced and its plan asserted, so that no change of the planner moves
the coverage.  Whole numbers: every entry of one form equals the other's, and
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


@pytest.mark.parametrize("scheme", [0, 1])
@pytest.mark.parametrize("s,R", [(1000, 5001), (10000, 3400)])
def test_per_step_chunks_over_a_whole_horizon(Bd, orc, s, R, scheme):
    """2,000-station DAG, T = 50: chunks of some 1,650 replications (64 MiB of
    state), the last one ragged."""
    run = W.scale_dag(s)
    n, E = run.net.n, run.net.nnz
    chunk = (64 << 20) // (4 * (n + 2 * E) + 32)
    assert R > 2 * chunk + 32 and R % (chunk // 32 * 32) != 0
    h = Bd.EulerNet(run.net)
    got = {}
    try:
        for form in (2, 1):
            h.set_option(Bd.OPT_FORM, form)
            assert h.plan(scheme, R)["form"] == form
            got[form] = h.simulate(scheme, run.dt, run.T, R, run.seed).cpu().numpy()
    finally:
        h.close()
    assert np.array_equal(got[1], got[2])
    rp = Bd.split_stats(got[2], n, R)["rep"]
    for r in (0, chunk + 40, R - 1):
        want = orc.simulate(run.net, scheme, run.dt, run.T, 1, run.seed, rep_begin=r)["rep"][0]
        assert np.array_equal(rp[r], want), r


@pytest.mark.parametrize("scheme", [0, 1])
def test_several_launches_of_tiles(Bd, scheme):
    """100-station DAG, 30,000 replications x 10,000 steps: a wave of tiles is
    over 1e10 updates, so no two share a launch of at most 2e10."""
    run = W.layered_dag()
    R, K = 30000, Bd.num_steps(run.dt, run.T)
    h = Bd.EulerNet(run.net)
    got = {}
    try:
        for form in (1, 2):
            h.set_option(Bd.OPT_FORM, form)
            p = h.plan(scheme, R)
            assert p["form"] == form
            if form == 1:
                assert 2e10 / 2 < run.net.n * p["tile_reps"] * p["grid"] * K < 2e10
                assert -(-R // p["tile_reps"]) > p["grid"]
            got[form] = h.simulate(scheme, run.dt, run.T, R, run.seed, rep_begin=7).cpu().numpy()
    finally:
        h.close()
    assert np.array_equal(got[1], got[2])
