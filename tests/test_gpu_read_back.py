"""State, moments and summaries read back in gene-major order through the staging
area: sizes whose results come back in one copy, sizes copied array by array, and
sizes whose arrays take several pieces; the FP64 form's state must survive a
set/get round trip bit for bit, and the summaries must be the formulas of the
moments that are read (§3.1), evaluated in the same FP64 operations."""
import numpy as np
import pytest

import paper_1606_06659_gb300 as fbs
from paper_1606_06659_gb300 import synthetic
from tests._pairs import STATE_KEYS

pytestmark = pytest.mark.gpu


def _data(N, G, L):
    X = synthetic.two_group_design(N) if L == 2 else np.ones((N, 1))
    d = synthetic.simulate(X, (2.0, 0.5)[:L], (1.0, 0.3)[:L], 0.2, 5.0, G, seed=N + G)
    d["priors"] = synthetic.default_priors(L)
    return d


@pytest.mark.parametrize("prec", [fbs.FBS_F64, fbs.FBS_F32])
@pytest.mark.parametrize("N,G,L", [(1, 2, 1), (5, 257, 2), (4, 2047, 2), (7, 5003, 2),
                                   (64, 2111, 2), (4, 70001, 2)])
def test_state_moments_and_summaries_round_trip(prec, N, G, L):
    d = _data(N, G, L)
    s = fbs.Sampler(d["y"], d["X"], d["h"], d["priors"], seed=1, precision=prec)
    rng = np.random.default_rng(G)
    st = {k: np.float32(rng.uniform(0.5, 1.5, np.shape(v))).astype(np.float64)
          for k, v in s.get_state().items() if k in STATE_KEYS}
    s.set_state(it=3, **st)
    got = s.get_state()
    for k in STATE_KEYS:
        assert np.array_equal(got[k], st[k]), k
    assert got["it"] == 3
    s.run(3, burnin=3)
    m = s.moments()
    assert m["count"] == 3
    st = s.get_state()
    e = s.estimates(eps=True)
    for v in ("eps", "beta", "gam", "phi"):
        mean, msq = m["mean_" + v], m["msq_" + v]
        sd = np.sqrt(np.maximum(msq - mean * mean, 0.0))
        assert np.array_equal(e["mean_" + v], mean), v
        # the device may fuse msq - mean^2; its rounding is at most 2^-53 of msq
        np.testing.assert_allclose(e["sd_" + v] ** 2, sd ** 2, rtol=1e-14,
                                   atol=float(np.abs(msq).max()) * 2.0 ** -51)
        np.testing.assert_allclose(e["lo_" + v], mean - fbs.Z95 * e["sd_" + v], rtol=1e-14,
                                   atol=float(np.abs(mean).max()) * 1e-15)
        np.testing.assert_allclose(e["hi_" + v], mean + fbs.Z95 * e["sd_" + v], rtol=1e-14,
                                   atol=float(np.abs(mean).max()) * 1e-15)
    again = s.get_state()
    for k in STATE_KEYS:
        assert np.array_equal(st[k], again[k]), k
    # reading between sweeps leaves the chain as it is
    t = fbs.Sampler(d["y"], d["X"], d["h"], d["priors"], seed=1, precision=prec)
    t.set_state(**{k: got[k] for k in STATE_KEYS}, it=3)
    t.run(5, burnin=3)
    s.run(2, burnin=3)
    a, b = s.get_state(), t.get_state()
    for k in STATE_KEYS:
        assert np.array_equal(a[k], b[k]), k
    s.close()
    t.close()


def test_summaries_into_new_arrays_cost_what_their_pages_cost():
    """Arrays whose pages were never touched: the call may take as long as into used
    ones and what the host takes to touch such pages, here with a factor of two,
    but not the several times that of pages faulted in by the copies."""
    import ctypes
    import mmap
    import time
    N, G = 32, 60000
    d = _data(N, G, 2)
    s = fbs.Sampler(d["y"], d["X"], d["h"], d["priors"], seed=1, precision=fbs.FBS_F32)
    s.run(4, burnin=2)

    def arrays():
        return [np.frombuffer(mmap.mmap(-1, G * N * 8), np.float64).reshape(G, N) for _ in range(4)]

    def call(out):
        o = fbs.EstimatesOut()
        o.z = 2.0
        for q, a in zip(("mean", "sd", "lo", "hi"), out):
            setattr(o, q + "_eps", a.ctypes.data_as(ctypes.POINTER(ctypes.c_double)))
        h = (ctypes.c_void_p * 1)(s.h)
        t = time.perf_counter()
        assert s.lib.fbs_estimates_pooled(1, h, ctypes.byref(o)) == 0
        return time.perf_counter() - t

    def fill(out):
        t = time.perf_counter()
        for a in out:
            a[:] = 1.0
        return time.perf_counter() - t

    used = arrays()
    call(used)
    host = min(fill(arrays()) for _ in range(5))
    again = min(call(used) for _ in range(5))
    times = []
    for _ in range(5):
        out = arrays()
        times.append(call(out))
        assert all(np.array_equal(a, b) for a, b in zip(out, used))
    assert min(times) < again + 2.0 * host, (min(times), again, host)
    s.close()
