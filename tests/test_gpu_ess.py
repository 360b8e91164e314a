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


def _write_trace(s, values):
    """values [rows][G][L] in place of the beta trace, which lies as [rows][L][G]
    doubles in the workspace that the sampler has from torch."""
    import torch
    have = np.ascontiguousarray(s.trace(beta=True)["beta"].transpose(0, 2, 1)).ravel()
    ws = s._ws[:s._ws.numel() // 8 * 8].view(torch.float64)
    host = ws.cpu().numpy()
    at = [i for i in np.flatnonzero(host[:host.size - have.size + 1] == have[0])
          if np.array_equal(host[i:i + have.size], have)]
    assert len(at) == 1
    new = np.ascontiguousarray(values.transpose(0, 2, 1)).ravel()
    ws[at[0]:at[0] + have.size] = torch.from_numpy(new).cuda()
    assert np.array_equal(s.trace(beta=True)["beta"], values)


def _ess_and_bound(x):
    """The effective sample size of x in extended precision, and how far an FP64 or
    55-bit form may be from it (u = 2^-53): the residuals carry the error m of the
    mean, their own rounding u |a| and 2^-55 of the largest magnitude M; a
    normalised autocovariance has seven more roundings (at lag 0 it is 1, whatever
    they are), the pair, the sum, tau and the division one each."""
    ld, u, n = np.longdouble, 2.0 ** -53, len(x)
    a = x.astype(ld) - x.astype(ld).sum() / n
    m = u * float(np.abs(x).sum())
    a2 = float((a * a).sum())
    fixed = 2.0 * 2.0 ** -55 * float(np.abs(a).max() * np.abs(a).sum()) / a2
    total, prev, err, k = ld(0), ld(np.inf), 0.0, 0
    while k + 1 < n:
        pair = ld(0)
        for j in (k, k + 1):
            p, q = a[:n - j], a[j:]
            r = (p * q).sum() / a2
            pair += r
            if j:
                err += ((2.0 * u * float(np.abs(p * q).sum()) + m * abs(float(p.sum() + q.sum()))
                         + n * m * m) / a2 + fixed
                        + float(abs(r)) * (9.0 * u + fixed + n * m * m / a2))
        if not pair > 0:
            break
        total, prev, k = total + min(pair, prev), min(pair, prev), k + 2
        err += u * float(prev + total)
    tau = -1 + 2 * total
    return float(n / tau), 2.0 * err / float(tau) + 2.0 * u


@pytest.mark.parametrize("rows", [250, 1295, 1296])
def test_beta_ess_of_series_of_a_wide_range(rows):
    """Series whose small values lie far below their largest one must keep as many
    bits as in FP64: noise with one value of 1e6, and the exponential of a series."""
    G, L = 40, 2
    d = synthetic.make_config(0, G=G)
    s = fbs.Sampler(d["y"], d["X"], d["h"], d["priors"], seed=rows, precision=fbs.FBS_F32,
                    trace_cap=rows, trace_beta=1)
    s.run(rows + 20, burnin=20, thin=1)
    rng = np.random.default_rng(rows)
    z = rng.normal(size=(rows, G, L))
    for t in range(1, rows):
        z[t] = 0.5 * z[t - 1] + z[t]
    z[rng.integers(0, rows, G), np.arange(G), 0] = 1e6
    z[:, :, 1] = np.exp(2.0 * z[:, :, 1])
    _write_trace(s, z)
    got = s.beta_ess()
    for g in range(G):
        for l in range(L):
            want, rel = _ess_and_bound(z[:, g, l])
            assert rel < (2e-15 if l == 0 else 1e-13)
            assert got[g, l] == pytest.approx(want, rel=rel), (g, l)
    s.close()
