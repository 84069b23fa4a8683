"""Per-step kernels after a larger call on the same handle (GPU): the state of
the larger call is kept, and a smaller call's customers and score sums use their
own stride.  Whole numbers and float64 sums in a fixed order: every entry equals
that of a new handle's call in the persistent form.
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


def _sojourn(Bd, h, scheme, R):
    import torch
    stats = torch.empty(Bd.stats_len(h.n, R), dtype=torch.int64, device="cuda")
    t = h.sojourn(scheme, 0.05, 2.0, R, 7, station=0, tau0=3, samples=5, stats=stats)
    return [t.cpu().numpy(), stats.cpu().numpy()]


def _grad(Bd, h, scheme, R):
    g = h.grad(scheme, 0.05, 2.0, R, 7, scores=True, stats=True)
    return [g[k].cpu().numpy() for k in ("grad", "value", "var", "scores", "stats")]


@pytest.mark.parametrize("call", [_sojourn, _grad])
@pytest.mark.parametrize("scheme", [0, 1])
def test_smaller_call_after_larger(Bd, call, scheme):
    net = W.random_small_dag(np.random.default_rng(3), 20, max_deg=3, m_range=(1, 9), ext_frac=0.5, lam_scale=20.0)
    h = Bd.EulerNet(net)
    try:
        h.set_option(Bd.OPT_FORM, 2)
        h.simulate(scheme, 0.05, 1.0, 600, 7)
        for R in (401, 33):
            f = Bd.EulerNet(net)
            try:
                f.set_option(Bd.OPT_FORM, 1)
                want = call(Bd, f, scheme, R)
            finally:
                f.close()
            for chunk in (-1, 96):
                h.set_option(Bd.OPT_HBM_CHUNK, chunk)
                for a, b in zip(call(Bd, h, scheme, R), want):
                    assert np.array_equal(a, b), (R, chunk)
            h.set_option(Bd.OPT_HBM_CHUNK, -1)
    finally:
        h.close()
