"""Direct-sampling statistics beyond the sizes of one tile: the autocorrelation's
exact sums on series whose products leave 128 bits, its lag and time tiles, and
a captured call.  References are plain FP64 sums over the same series (another
order: 1e-10 relative, as against the oracle)."""
import numpy as np
import pytest
import torch

pytestmark = pytest.mark.gpu


@pytest.fixture(scope="module")
def L():
    from paper_2005_09323_gb300 import build, lbmrare
    build.build()
    lbmrare.lib()
    return lbmrare


class Series:
    """an ensemble whose drag history is the given series"""

    def __init__(self, L, d, stream=None):
        self.L, (n, steps) = L, d.shape
        self.e = L.lbm_ensemble_create(L.config(16, 4, tau=0.8, max_steps=steps), n, 1,
                                       stream or torch.cuda.current_stream())
        L.lbm_ensemble_step(self.e, steps)
        L.lbm_ensemble_set_drag(self.e, 0, steps, d)

    def __enter__(self):
        return self.e

    def __exit__(self, *a):
        self.L.lbm_ensemble_destroy(self.e)


def reference(d, lags):
    x = d - d.mean()
    var = np.mean(x * x)
    n, m = x.shape
    return np.array([np.dot(x[:, :m - k].ravel(), x[:, k:].ravel()) / (n * (m - k)) / var for k in lags])


def sine(n, steps, period):
    t = np.arange(steps)[None, :] + np.linspace(0, period, n, endpoint=False)[:, None]
    return 0.4 + 0.03 * np.sin(2 * np.pi * t / period)


def two_level(n, steps, period):
    return 0.4 + 0.03 * np.where(sine(n, steps, period) >= 0.4, 1.0, -1.0)


# sums of 2.2 and 4.5 times 2^127 in units of the fixed-point products; the third with
# more than 512 tasks (clone, 512 steps) to a thread.  The correlation crosses zero at a
# quarter period
@pytest.mark.parametrize("form,period,tau_c,n,steps,max_lag", [(sine, 487, 122, 128, 20000, 600),
                                                               (two_level, 498, 125, 128, 20000, 600),
                                                               (two_level, 498, 125, 400, 40000, 16383)])
def test_autocorrelation_of_long_full_scale_series(L, form, period, tau_c, n, steps, max_lag):
    d = form(n, steps, period)
    lags = [k for k in (0, 1, 60, tau_c - 1, tau_c, 250, 511, 512, 600, 8192, 16383) if k <= max_lag]
    with Series(L, d) as e:
        c = torch.zeros(max_lag + 1, dtype=torch.float64, device="cuda")
        assert L.lbm_drag_autocorrelation(e, 0, steps, max_lag, c) == tau_c
    got = c.cpu().numpy()
    assert abs(got[0] - 1.0) <= 1e-10
    assert np.allclose(got[lags], reference(d, lags), rtol=1e-10, atol=1e-12)


# the edges of the 512-lag and 512-step tiles, one series of one step more than its
# lags, and more (clone, 512 steps) tasks than splits of the sum
@pytest.mark.parametrize("n,steps,t0,max_lag", [(3, 1025, 0, 512), (3, 1024, 1, 511), (2, 1600, 37, 1024),
                                                (1, 700, 0, 699), (300, 4100, 3, 600), (700, 520, 0, 2)])
def test_autocorrelation_at_tile_edges(L, n, steps, t0, max_lag):
    from tests import seeded_inputs as si
    d = si.drag_series(n, steps, 9, rho=0.97)
    lags = sorted({k for k in (0, 1, 2, 3, 4, 127, 128, 510, 511, 512, 513, 1023, 1024, max_lag - 1, max_lag)
                   if k <= max_lag})
    with Series(L, d) as e:
        c = torch.zeros(max_lag + 1, dtype=torch.float64, device="cuda")
        L.lbm_drag_autocorrelation(e, t0, steps, max_lag, c)
    assert np.allclose(c.cpu().numpy()[lags], reference(d[:, t0:], lags), rtol=1e-10, atol=1e-12)


def test_captured_autocorrelation_outlives_the_workspace(L):
    """A call captured after a warm-up, then a larger call that replaces the
    ensemble's workspace, then the captured work replayed on a changed series:
    the same bits as a direct call, and the larger call's result untouched"""
    rng = np.random.default_rng(3)
    n, steps, lag = 4, 3000, 40
    d = rng.normal(0.4, 0.01, (n, steps))
    s = torch.cuda.Stream()
    with Series(L, d, s) as e:
        small, direct = (torch.zeros(lag + 1, dtype=torch.float64, device="cuda") for _ in range(2))
        large = torch.zeros(2900, dtype=torch.float64, device="cuda")
        torch.cuda.synchronize()
        call = L.lib().lbm_drag_autocorrelation
        assert call(e, 0, 600, lag, small.data_ptr(), None) == 0
        s.synchronize()
        g = torch.cuda.CUDAGraph()
        with torch.cuda.graph(g, stream=s):
            assert call(e, 0, 600, lag, small.data_ptr(), None) == 0
        L.lbm_drag_autocorrelation(e, 0, steps, 2899, large)
        before = large.clone()
        d[:, :600] = rng.normal(0.4, 0.02, (n, 600))
        L.lbm_ensemble_set_drag(e, 0, steps, d)
        small.zero_()
        torch.cuda.synchronize()
        with torch.cuda.stream(s):
            for _ in range(2):
                g.replay()
        s.synchronize()
        L.lbm_drag_autocorrelation(e, 0, 600, lag, direct)
        assert torch.equal(small, direct) and float(direct[0]) != 0.0
        assert torch.equal(large, before)
        del g


@pytest.mark.parametrize("window,t_begin", [(1000, 0), (7, 3), (65, 69000)])
def test_scores_of_a_series_longer_than_the_block_table(L, window, t_begin):
    """trailing means of 70000 steps: the opening sums' blocks hold 35 steps there, 32
    below 65537 (bounds as for the short series: 1e-11)"""
    rng = np.random.default_rng(5)
    d = 0.4 + np.cumsum(rng.normal(0, 1e-4, (2, 70000)), axis=1)
    with Series(L, d) as e:
        q = torch.zeros(2, dtype=torch.float64, device="cuda")
        L.lbm_ensemble_scores(e, window, t_begin, 70000, q)
        got = q.cpu().numpy()
    s = np.concatenate([np.zeros((2, 1)), np.cumsum(d[:, t_begin:].astype(np.longdouble), axis=1)], axis=1)
    ref = ((s[:, window:] - s[:, :-window]).max(axis=1) / window).astype(np.float64)
    assert np.allclose(got, ref, rtol=1e-11, atol=1e-14)
