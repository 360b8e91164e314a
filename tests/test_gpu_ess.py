"""fbs_beta_ess on the device against the oracle's sequential FP64 form, at the
edges of the kernel's splits: few rows, rows that are no multiple of the lags of
a round, the row counts at which fewer series share a block, the traces that
take one thread per series, and series that never move.

Tolerance: a sum of n FP64 products carries at most n 2^-53 of the sum of their
magnitudes, so a normalised autocovariance n 2^-53; summed over at most n lags
and doubled, n^2 2^-52 relative to the series' tau >= 1 (n = 5001: 5.6e-9)."""
import numpy as np
import pytest

import oracle
import paper_1606_06659_gb300 as fbs
from paper_1606_06659_gb300 import synthetic

pytestmark = pytest.mark.gpu


def _check(s, rows, n_series=60):
    tr = s.trace(beta=True)["beta"]
    assert tr.shape[0] == rows
    got = s.beta_ess()
    G, L = got.shape
    rng = np.random.default_rng(rows)
    for i in np.unique(np.r_[0, G * L - 1, rng.integers(0, G * L, n_series)]):
        g, l = divmod(int(i), L)
        want = oracle.ess(np.ascontiguousarray(tr[:, g, l]))
        assert got[g, l] == pytest.approx(want, rel=max(rows * rows * 2.0 ** -52, 1e-12)), (g, l)


@pytest.mark.parametrize("rows,G", [(4, 37), (5, 1301), (16, 1301), (17, 609), (250, 1301),
                                    (1000, 1301), (1403, 1301), (1404, 1301), (2938, 700),
                                    (5000, 40), (5001, 40)])
def test_beta_ess_equals_the_sequential_form(rows, G):
    d = synthetic.make_config(0, G=G)
    s = fbs.Sampler(d["y"], d["X"], d["h"], d["priors"], seed=rows, precision=fbs.FBS_F32,
                    trace_cap=rows, trace_beta=1)
    s.run(rows + 20, burnin=20, thin=1)
    _check(s, rows)
    s.close()


def test_beta_ess_of_series_that_never_move():
    d = synthetic.make_config(0, G=90)
    s = fbs.Sampler(d["y"], d["X"], d["h"], d["priors"], seed=3, precision=fbs.FBS_F32,
                    trace_cap=77, trace_beta=1, shrink_max=0)
    s.run(77, burnin=0, thin=1)
    assert np.ptp(s.trace(beta=True)["beta"], axis=0).max() == 0.0
    _check(s, 77, 180)
    s.close()


@pytest.mark.parametrize("rows,G", [(64, 31), (250, 503), (1000, 503), (1295, 487), (1296, 487),
                                    (8000, 31), (8001, 31)])
def test_beta_ess_of_series_that_mix_slowly(rows, G):
    """Series that end after a few dozen to hundreds of lags: rounds with few of them left."""
    d = synthetic.make_config(1, G=G)
    s = fbs.Sampler(d["y"], d["X"], d["h"], d["priors"], seed=rows, precision=fbs.FBS_F32,
                    trace_cap=rows, trace_beta=1)
    s.run(rows + 200, burnin=200, thin=1)
    _check(s, rows, 120)
    s.close()
