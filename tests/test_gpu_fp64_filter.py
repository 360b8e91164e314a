"""The FP64 slice updates whose comparisons are decided in FP32 where an error
bound allows: lockstep with the oracle, element by element and with equal
evaluation counts, where the bound could go wrong (many value classes, values
far from one, widths far too small and far too large, step-out and shrinkage
limits at and near zero, counts from 0 to 2^30, tiny and huge gamma_g), and the
one-launch sweep on caller-owned arrays against fbs_run over the sizes of its
blocks."""
import numpy as np
import pytest

import paper_1606_06659_gb300 as fbs
from paper_1606_06659_gb300 import synthetic
from tests._pairs import (ALL_SLICE_KEYS, ATOL, RTOL, assert_state_close, close, make_pair,
                          sync_gpu_to_oracle)
from tests.test_gpu_parity import COUNTS

pytestmark = pytest.mark.gpu


def _design(kind, N):
    one = np.ones(N)
    if kind == "one":
        return one[:, None]
    if kind == "three":
        return np.stack([one, np.array([0.5, 2.0, -1.5])[np.arange(N) % 3]], axis=1)
    if kind == "eight":
        v = np.array([0.1, -0.2, 3.0, 1.0, -1.0, 0.75, -2.5, 0.3])
        return np.stack([one, np.where(np.arange(N) % 2 == 0, 1.0, -1.0), v[np.arange(N) % 8]],
                        axis=1)
    return synthetic.two_group_design(N)


def _data(kind, N, G, big=False):
    X = _design(kind, N)
    L = X.shape[1]
    d = synthetic.simulate(X, (2.0, 0.3, -0.1)[:L], (1.5, 0.3, 0.2)[:L], 0.2, 3.0, G, seed=N + G)
    d["priors"] = synthetic.default_priors(L)
    if big:
        d["y"] = d["y"].copy()
        d["y"][: G // 4] = 0
        d["y"][G // 4: G // 2] = 2 ** 30
        d["y"][G // 2: 3 * G // 4] *= 1000
    return d


@pytest.mark.parametrize("kind,N,G,big,opt", [
    ("two", 8, 300, True, {}),
    ("three", 9, 257, False, {}),
    ("eight", 16, 300, True, {}),
    ("two", 6, 300, True, dict(w0=1e-4)),
    ("eight", 17, 200, False, dict(w0=2e4)),
    ("two", 6, 200, False, dict(step_out_max=0)),
    ("two", 6, 200, False, dict(step_out_max=1, shrink_max=2)),
    ("three", 6, 200, False, dict(step_out_max=5000, w0=1e-3)),
    ("two", 6, 300, True, dict(all_slice=1)),
    ("eight", 8, 200, False, dict(all_slice=1, w0=50.0)),
    ("two", 6, 200, False, dict(all_slice=1, w0=1e-4)),
])
def test_lockstep(kind, N, G, big, opt):
    g, o = make_pair(_data(kind, N, G, big), seed=12345, **opt)
    o.init_default()
    o.set_opts(burnin=2, tune_start=1)
    for it in range(1, 4):
        sync_gpu_to_oracle(g, o, it - 1)
        c0, o0 = g.counters(), o.counters_dict()
        g.run(1, burnin=2, thin=1)  # get_state waits; sync would report the capped updates
        o.sweep()
        assert_state_close(g.get_state(), o.get_state(), keys=ALL_SLICE_KEYS, where=f"sweep {it}")
        c1, o1 = g.counters(), o.counters_dict()
        for k in COUNTS:
            assert c1[k] - c0[k] == o1[k] - o0[k], (it, k)


@pytest.mark.parametrize("kind,N,G", [("one", 1, 2), ("two", 5, 33), ("three", 9, 127),
                                      ("eight", 23, 128), ("two", 64, 129), ("eight", 16, 1201)])
def test_noalloc_equals_run(kind, N, G):
    import torch
    d = _data(kind, N, G)
    L = d["X"].shape[1]
    s = fbs.Sampler(d["y"], d["X"], d["h"], d["priors"], seed=8)
    st = s.get_state()

    def dev(a):
        return torch.from_numpy(np.ascontiguousarray(np.asarray(a).T)).cuda()

    arr = {k: dev(st[k]) for k in ("eps", "w_eps", "waux_eps", "beta", "w_beta", "waux_beta", "gam")}
    arr["y"] = dev(d["y"].astype(np.int32))
    arr["T"] = dev(d["y"].astype(np.float64) @ d["X"])
    arr["hyp"] = dev(np.concatenate([st["phi"], st["w_nu"], st["waux_nu"]]))
    for k, shape in (("eps", (N, G)), ("beta", (L, G)), ("gam", (G,)), ("phi", (2 * L + 2,))):
        arr["m_" + k] = torch.zeros(shape, dtype=torch.float64, device="cuda")
        arr["q_" + k] = torch.zeros(shape, dtype=torch.float64, device="cuda")
    status = torch.zeros(1 + fbs.NUM_COUNTERS, dtype=torch.int64, device="cuda")
    evals = 0
    for it in range(1, 6):
        fbs.sweep_noalloc(d["X"], d["h"], d["priors"], seed=8, it=it, burnin=3,
                          n_mom=max(0, it - 4), stream=torch.cuda.current_stream().cuda_stream,
                          G=G, status=status.data_ptr(), **{k: v.data_ptr() for k, v in arr.items()})
        evals += int(status[1].item())
    s.run(5, burnin=3)
    got, m, c = s.get_state(), s.moments(), s.counters()
    assert evals == c["evals_eps"]
    for k in ("eps", "w_eps", "waux_eps", "beta", "w_beta", "waux_beta", "gam"):
        assert close(arr[k].cpu().numpy().T, got[k], RTOL, ATOL).all(), k
    for k in ("eps", "beta", "gam", "phi"):
        assert close(arr["m_" + k].cpu().numpy().T, m["mean_" + k], RTOL, ATOL).all(), k
        assert close(arr["q_" + k].cpu().numpy().T, m["msq_" + k], RTOL, ATOL).all(), k
    assert close(arr["hyp"].cpu().numpy()[: 2 * L + 2], got["phi"], RTOL, ATOL).all()
    s.close()


def test_noalloc_rounds_the_squares_of_eps():
    """The second moments of eps fold in the square rounded to FP64: with one draw
    before it the weight of the next is 1/2, so that everything else is exact but
    the subtraction and the final sum."""
    import torch
    d = _data("two", 9, 1501)
    L, (G, N) = 2, d["y"].shape
    s = fbs.Sampler(d["y"], d["X"], d["h"], d["priors"], seed=8)
    st = s.get_state()
    s.close()

    def dev(a):
        return torch.from_numpy(np.ascontiguousarray(np.asarray(a).T)).cuda()

    arr = {k: dev(st[k]) for k in ("eps", "w_eps", "waux_eps", "beta", "w_beta", "waux_beta", "gam")}
    arr["y"] = dev(d["y"].astype(np.int32))
    arr["T"] = dev(d["y"].astype(np.float64) @ d["X"])
    arr["hyp"] = dev(np.concatenate([st["phi"], st["w_nu"], st["waux_nu"]]))
    for k, shape in (("eps", (N, G)), ("beta", (L, G)), ("gam", (G,)), ("phi", (2 * L + 2,))):
        arr["m_" + k] = torch.zeros(shape, dtype=torch.float64, device="cuda")
        arr["q_" + k] = torch.zeros(shape, dtype=torch.float64, device="cuda")
    q = np.zeros((N, G))
    for it in range(1, 3):
        fbs.sweep_noalloc(d["X"], d["h"], d["priors"], seed=8, it=it, burnin=0, n_mom=it - 1,
                          stream=torch.cuda.current_stream().cuda_stream, G=G,
                          **{k: v.data_ptr() for k, v in arr.items()})
        x = arr["eps"].cpu().numpy()
        q = q + (x * x - q) / it
        assert np.array_equal(arr["q_eps"].cpu().numpy(), q), it


@pytest.mark.parametrize("kind", ["three", "eight"])
def test_lockstep_above_the_genes_of_split_blocks(kind):
    """More genes than the blocks with gamma on a second warp hold at once: the
    one-warp blocks, with columns of three and eight value classes."""
    import torch
    G = 32 * 6 * torch.cuda.get_device_properties(0).multi_processor_count + 33
    g, o = make_pair(_data(kind, 9, G), seed=7)
    o.init_default()
    o.set_opts(burnin=1, tune_start=0)
    for it in range(1, 3):
        sync_gpu_to_oracle(g, o, it - 1)
        c0, o0 = g.counters(), o.counters_dict()
        g.run(1, burnin=1, thin=1)
        o.sweep()
        assert_state_close(g.get_state(), o.get_state(), where=f"sweep {it}")
        c1, o1 = g.counters(), o.counters_dict()
        for k in COUNTS:
            assert c1[k] - c0[k] == o1[k] - o0[k], (it, k)
