"""Handles of different sizes side by side: the limit of a kernel's dynamic shared
memory belongs to the process, so a handle that sets it to its own need would make
the launches of a larger one fail.  Every pair needs more than the 48 KB that no
limit has to be set for; the larger handle must run as if it were alone."""
import threading

import numpy as np
import pytest

import paper_1606_06659_gb300 as fbs
from paper_1606_06659_gb300 import synthetic

pytestmark = pytest.mark.gpu

KEYS = ("eps", "beta", "gam", "phi", "w_eps", "w_beta")


def _data(N, G=300, levels=8):
    """A treatment and a dose of `levels` values: up to 16 distinct rows of X."""
    X = synthetic.two_group_design(N)
    if levels:
        dose = np.array([0.0, 0.25, 0.5, 1.0, 1.5, 2.0, 3.0, -1.0])[np.arange(N) % levels]
        X = np.column_stack([X, dose])
    L = X.shape[1]
    d = synthetic.simulate(X, (3.0, 0.0, 0.0)[:L], (1.5, 0.3, 0.1)[:L], 0.1, 3.0, G, seed=N)
    d["priors"] = synthetic.default_priors(L)
    return d


def _sampler(d, form, seed=5, **kw):
    prec = fbs.FBS_F64 if form == "f64" else fbs.FBS_F32
    s = fbs.Sampler(d["y"], d["X"], d["h"], d["priors"], seed=seed, precision=prec, block=128, **kw)
    if form in ("move", "net"):
        L = d["X"].shape[1]
        rng = np.random.default_rng(1)
        s.proposal_params(set_to=(0.05 * rng.normal(size=fbs.proposal_param_count(L)))
                          .astype(np.float32))
        s.proposal_fused(form == "net")
    return s


def _run(s, form, sweeps):
    if form in ("move", "net"):
        s.proposal_calibrate(4, burnin=1000, min_accept=0.0)
    s.run(sweeps, burnin=1000)
    s.sync()
    return s.get_state()


@pytest.mark.parametrize("sweeps", [5, 100])  # direct launches; the capture of a segment
@pytest.mark.parametrize("form,small,large", [
    ("f32", (22, 8), (40, 8)),
    ("f32", (64, 0), (64, 8)),  # equal N: only the number of distinct rows differs
    ("move", (22, 8), (40, 8)),
    ("net", (22, 8), (40, 8)),
    ("f64", (30, 0), (64, 0)),
])
def test_a_smaller_handle_leaves_a_larger_one_running(form, small, large, sweeps):
    d, e = _data(large[0], levels=large[1]), _data(small[0], levels=small[1])
    a = _sampler(d, form)
    want = _run(a, form, sweeps)
    a.close()
    a = _sampler(d, form)
    b = _sampler(e, form)
    _run(b, form, 3)
    got = _run(a, form, sweeps)
    _run(b, form, 3)
    for k in KEYS:
        assert np.array_equal(got[k], want[k]), k
    a.close()
    b.close()


def test_a_smaller_batch_leaves_a_larger_one_running():
    sets = [_data(40), _data(6, levels=0)], [_data(22), _data(5, levels=0)]
    want = []
    for _ in range(2):
        a = fbs.BatchSampler(sets[0], seeds=[1, 2])
        b = fbs.BatchSampler(sets[1], seeds=[3, 4]) if want else None
        a.run(5, burnin=1000)
        a.sync()
        want.append([v.get_state() for v in a.views])
        if b is not None:
            b.run(5, burnin=1000)
            b.sync()
            b.close()
        a.close()
    for x, y in zip(*want):
        for k in KEYS:
            assert np.array_equal(x[k], y[k]), k


def _threads(work):
    """work[i] run over and over by a thread each; the first error of any."""
    errors = []

    def loop(f, n):
        try:
            for _ in range(n):
                f()
        except Exception as e:  # noqa: BLE001 (handed to the test)
            errors.append(e)

    threads = [threading.Thread(target=loop, args=w) for w in work]
    for t in threads:
        t.start()
    for t in threads:
        t.join()
    if errors:
        raise errors[0]


def test_network_kernels_of_threads():
    a, b = (_sampler(_data(N), "net") for N in (40, 22))
    for s in (a, b):
        s.proposal_calibrate(4, burnin=10 ** 6, min_accept=0.0)

    def work(s):
        s.run(20, burnin=10 ** 6)
        s.sync()

    _threads([(lambda: work(a), 100), (lambda: work(b), 100)])
    a.close()
    b.close()


def _collected(X, seed):
    L = X.shape[1]
    d = synthetic.simulate(X, (3.0,) + (0.0,) * (L - 1), (1.5,) + (0.3,) * (L - 1), 0.1, 3.0, 300,
                           seed=L)
    s = fbs.Sampler(d["y"], X, d["h"], synthetic.default_priors(L), seed=seed,
                    precision=fbs.FBS_F32)
    s.run(20, burnin=1000)
    s.proposal_collect(10, burnin=1000)
    return s


@pytest.mark.parametrize("other", ["train", "gradient"])
def test_training_of_fewer_columns_between_two_training_calls(other):
    """A handle keeps its training buffers; the kernel's limit for its L = 5 must
    outlast another handle's training, or a gradient call, at L = 2."""
    def train(s):
        return s.proposal_train(epochs=2, batch=512, lr=1e-3, seed=3)

    X = synthetic.paper_design(4)
    s = _collected(X, 7)
    want = train(s), train(s), s.proposal_params()
    s.close()
    s = _collected(X, 7)
    first = train(s)
    if other == "train":
        t = _collected(synthetic.two_group_design(8), 8)
        train(t)
        t.close()
    else:
        rng = np.random.default_rng(2)
        fbs.proposal_loss_grad((0.1 * rng.normal(size=fbs.proposal_param_count(2)))
                               .astype(np.float32), 2, rng.normal(size=(40, 9)),
                               rng.normal(size=(40, 2)))
    assert (first, train(s)) == want[:2]
    assert np.array_equal(s.proposal_params(), want[2])
    s.close()


@pytest.mark.parametrize("rows", [(1290, 8), (4000, 1300)])  # four and two series per block
def test_ess_of_traces_of_different_lengths_in_several_threads(rows):
    """One long trace beside six short ones, whose calls come between its own."""
    chains = []
    for i, n in enumerate((rows[0],) + 6 * (rows[1],)):
        d = synthetic.make_config(0, G=2, seed=i)
        s = fbs.Sampler(d["y"], d["X"], d["h"], d["priors"], seed=n, precision=fbs.FBS_F32,
                        trace_cap=n, trace_beta=1)
        s.run(n + 20, burnin=20, thin=1)
        s.sync()
        chains.append((s, s.beta_ess()))

    def work(s, want):
        assert np.array_equal(s.beta_ess(), want)

    _threads([(lambda c=c: work(*c), 3000) for c in chains])
    for s, _ in chains:
        s.close()
