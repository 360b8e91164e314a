"""The work whose speed is measured: calls a user of the sampler makes through its
public entry points, at sizes from the smallest dataset to the largest one the
repository configures.

A case is a dict with a "kind":

  chain    a running chain (tuned, past its burn-in) continued by a window of
           sweeps, then the posterior summaries or the whole state read back
  job      a whole small job from host counts: create, run, summaries
  batch    many uneven datasets swept together, each dataset's summaries read
  noalloc  one sweep on arrays the caller owns
  train    one call that trains the learned proposal on collected pairs
  grad     the proposal network's loss and gradient on a batch
  summary  what is computed once at the end of a job: effective sample sizes,
           Gelman-Rubin factors and pooled estimates of two traced chains

Sizes are those of the repository's configurations (N=4 G=1000 L=2; N=16
G=40000 L=5; N=32 G=200000 L=5; datasets of N in 4..32, G in 1e3..1e5) and odd
sizes between and below them.
"""
from __future__ import annotations

import math

import numpy as np
import torch

import paper_1606_06659_gb300 as fbs
from paper_1606_06659_gb300 import synthetic

# Sweeps that tune the slice widths before a chain is handed over.
TUNE = 200
H = 64  # hidden units of the proposal network


# ------------------------------------------------------------------ cases

def listed():
    return [
        # the smallest interactive use: one sweep of a few hundred genes, then
        # the whole state (a program that inspects or checkpoints every sweep)
        dict(name="step_small", kind="chain", form="f32", design="two", N=5, G=257, sweeps=1,
             read="state"),
        # the repository's smallest configuration as a whole FP64 job
        dict(name="job_tiny_f64", kind="job", form="f64", design="two", N=4, G=1000, iters=1000),
        # a mid-size FP32 chain with a covariate of several levels (more distinct
        # rows of X than the per-row sums hold), odd sizes, checkpointed
        dict(name="chain_covariate_f32", kind="chain", form="f32", design="covariate", N=22,
             G=9973, sweeps=100, read="state"),
        # the paper's workload in its three forms: FP64 (the default form), FP32, and
        # FP32 with the learned proposal (the benchmark's headline)
        dict(name="paper_f64", kind="chain", form="f64", design="paper", N=16, G=40000,
             sweeps=20, read="estimates"),
        dict(name="paper_f32", kind="chain", form="f32", design="paper", N=16, G=40000,
             sweeps=300, read="estimates"),
        dict(name="paper_learned", kind="chain", form="learned", design="paper", N=16, G=40000,
             sweeps=300, read="estimates"),
        # the paper's own choice of slice updates for every non-normal conditional
        dict(name="all_slice_f64", kind="chain", form="all_slice", design="paper", N=12, G=12345,
             sweeps=20, read="estimates"),
        # the precision-stress configuration, the largest dataset
        dict(name="stress_f32", kind="chain", form="f32", design="paper", N=32, G=200000,
             sweeps=100, read="estimates"),
        # uneven datasets in one set of launches
        dict(name="batch_uneven", kind="batch", sets=24, min_G=1000, max_G=30000, sizes=1,
             sweeps=100, top=False),
        # a caller that may not allocate, one FP64 sweep at a time
        dict(name="noalloc_sweep", kind="noalloc", design="paper", N=16, G=20011),
        # training the learned proposal inside a job
        dict(name="train_epoch", kind="train", N=16, G=40000, collect=25, batch=8192),
        # the end of a job: ESS of every beta, Gelman-Rubin, pooled summaries
        dict(name="end_of_job", kind="summary", N=16, G=6007, rows=1000),
    ]


def _log_int(rng, lo, hi):
    return int(round(math.exp(rng.uniform(math.log(lo), math.log(hi)))))


def draw(rng):
    kind = rng.choice(["chain"] * 6 + ["job", "batch", "noalloc", "train", "grad", "summary"])
    if kind == "chain":
        form = rng.choice(["f32", "f32", "learned", "f64", "all_slice"])
        design = rng.choice(["two", "paper", "paper", "covariate"])
        N = 4 * rng.randint(2, 8) if design == "paper" else rng.randint(6, 32)
        G = _log_int(rng, 200, 60000)
        work = {"f32": 3e8, "learned": 1.5e8, "f64": 1.2e7, "all_slice": 1.2e7}[form]
        sweeps = max(1, min(300, int(rng.uniform(0.1, 1.0) * work / (N * G))))
        return dict(kind="chain", form=form, design=design, N=N, G=G, sweeps=sweeps,
                    read=rng.choice(["estimates", "estimates", "state"]))
    if kind == "job":
        return dict(kind="job", form=rng.choice(["f64", "f32"]), design="two", N=rng.randint(4, 9),
                    G=_log_int(rng, 150, 3000), iters=100 * rng.randint(2, 12))
    if kind == "batch":
        return dict(kind="batch", sets=rng.randint(2, 24), min_G=_log_int(rng, 200, 1500),
                    max_G=_log_int(rng, 2000, 30000), sizes=rng.randint(1, 1000),
                    sweeps=rng.randint(20, 100), top=rng.random() < 0.5)
    if kind == "noalloc":
        design = rng.choice(["two", "paper", "covariate"])
        N = 4 * rng.randint(2, 8) if design == "paper" else rng.randint(6, 32)
        return dict(kind="noalloc", design=design, N=N, G=_log_int(rng, 300, 30000))
    if kind == "train":
        return dict(kind="train", N=4 * rng.randint(2, 5), G=_log_int(rng, 3000, 30000),
                    collect=rng.randint(5, 25), batch=1024 * rng.randint(2, 12))
    if kind == "grad":
        return dict(kind="grad", L=rng.choice([2, 3, 5, 8]), B=_log_int(rng, 40, 16000))
    return dict(kind="summary", N=4 * rng.randint(2, 5), G=_log_int(rng, 300, 8000),
                rows=rng.randint(200, 1000))


# ------------------------------------------------------------------ inputs

PARAMS = {2: ((3.0, 0.0), (1.5, 0.3)), 3: ((3.0, 0.0, 0.0), (1.5, 0.3, 0.1)),
          5: ((4.0, 0.0, 0.0, 0.0, 0.0), (2.0, 0.5, 0.3, 0.2, 0.2))}


def _design(name, N):
    if name == "paper":
        return synthetic.paper_design(N // 4)
    X = synthetic.two_group_design(N)
    if name == "covariate":  # a dose of up to eight levels beside the treatment
        dose = np.array([0.0, 0.25, 0.5, 1.0, 1.5, 2.0, 3.0, -1.0])[np.arange(N) % 8]
        X = np.column_stack([X, dose])
    return X


def _simulate(X, G, seed):
    """Counts drawn from the model on the GPU (the generator of
    ``synthetic.simulate`` with torch's random numbers) and the values behind them."""
    N, L = X.shape
    theta, sigma = PARAMS[L]
    gen = torch.Generator(device="cuda").manual_seed(int(seed))
    f = dict(device="cuda", dtype=torch.float64)

    def normal(*shape):
        return torch.randn(*shape, generator=gen, **f)

    nu, tau = 3.0, 0.1
    h = 0.1 * normal(N)
    # 1/gamma_g ~ Gamma(nu/2, rate nu tau/2) with nu = 3: a chi-square of 3 degrees
    gam = nu * tau / normal(G, 3).square().sum(1)
    eps = normal(G, N) * gam.sqrt()[:, None]
    beta = normal(G, L) * torch.tensor(sigma, **f) + torch.tensor(theta, **f)
    eta = h + eps + beta @ torch.tensor(X, **f).T
    y = torch.poisson(eta.exp().clamp(max=float(2 ** 30)), generator=gen)
    return {"y": y.to(torch.int32).cpu().numpy(), "X": X, "h": h.cpu().numpy(),
            "priors": synthetic.default_priors(L), "eps": eps, "beta": beta, "gam": gam}


def _sampler(d, form, seed, **kw):
    kw.setdefault("precision", fbs.FBS_F64 if form in ("f64", "all_slice") else fbs.FBS_F32)
    if form == "all_slice":
        kw["all_slice"] = 1
    return fbs.Sampler(d["y"], d["X"], d["h"], d["priors"], seed=seed, **kw)


def _batch_sizes(case):
    """(design, N, G) of every dataset: N uniform on 4..32, G log-uniform, the
    paper's design for half of them (the three-level model wants one L for all)."""
    rng = np.random.default_rng(case["sizes"])
    out = []
    for _ in range(case["sets"]):
        N = int(rng.integers(4, 33))
        G = int(np.exp(rng.uniform(np.log(case["min_G"]), np.log(case["max_G"]))))
        paper = rng.integers(0, 2) == 1 and not case["top"]
        out.append(("paper", max(8, N // 4 * 4), G) if paper else ("two", N, G))
    return out


# ------------------------------------------------------------------ prepare

def prepare(case, seed):
    kind = case["kind"]
    state = dict(case=case, seed=seed)
    if kind in ("chain", "job", "noalloc"):
        d = _simulate(_design(case["design"], case["N"]), case["G"], seed)
    if kind == "chain":
        s = _sampler(d, case["form"], seed)
        burnin = TUNE
        s.run(TUNE, burnin=burnin, thin=10)
        if case["form"] == "learned":  # the proposal is trained and calibrated in the burn-in
            burnin = 1 << 20
            s.proposal_collect(max(4, min(25, -(-200000 // case["G"]))), burnin=burnin, thin=2)
            s.proposal_train(epochs=4, batch=8192, lr=3e-3, seed=seed)
            s.proposal_calibrate(40, burnin=burnin, min_accept=0.01)
            burnin = s.get_state()["it"]
        s.run(100, burnin=burnin, thin=10)  # the first segment of the chain proper
        s.sync()
        state.update(s=s, burnin=burnin)
    elif kind == "job":
        state.update(d={k: d[k] for k in ("y", "X", "h", "priors")})
    elif kind == "batch":
        sets = [_simulate(_design(design, N), G, seed * 1000 + i)
                for i, (design, N, G) in enumerate(_batch_sizes(case))]
        b = fbs.BatchSampler(sets, seeds=[seed + i for i in range(len(sets))])
        if case["top"]:
            b.three_level(e=10.0, a_b=1.0, b_b=1.0, seed=seed)
        b.run(TUNE, burnin=TUNE, thin=10)
        b.sync()
        state.update(b=b)
    elif kind == "noalloc":
        state.update(_noalloc_arrays(d, seed))
    elif kind == "train":
        d = _simulate(_design("paper", case["N"]), case["G"], seed)
        s = _sampler(d, "f32", seed)
        s.run(TUNE, burnin=1 << 20, thin=10)
        s.proposal_collect(case["collect"], burnin=1 << 20, thin=2)
        s.sync()
        state.update(s=s)
    elif kind == "grad":
        state.update(_grad_inputs(case["L"], case["B"], seed))
    else:
        d = _simulate(_design("paper", case["N"]), case["G"], seed)
        chains = [_sampler(d, "f32", seed, chain=c, trace_cap=case["rows"], trace_beta=1)
                  for c in range(2)]
        for s in chains:
            s.run(TUNE + case["rows"], burnin=TUNE, thin=1)
            s.sync()
        state.update(chains=chains)
    return state


def _noalloc_state(d, seed):
    """A tuned-looking state around the values the counts were drawn from: widths
    of the order of the conditional standard deviations."""
    N, L = d["X"].shape
    y = torch.tensor(d["y"], device="cuda", dtype=torch.float64)
    gam = d["gam"]
    theta, sigma = PARAMS[L]
    prec = y + 1.0
    st = {"eps": d["eps"].T, "w_eps": (2.0 / (prec + 1.0 / gam[:, None]).sqrt()).T,
          "beta": d["beta"].T}
    X = torch.tensor(d["X"], device="cuda", dtype=torch.float64)
    s2 = torch.tensor(sigma, device="cuda", dtype=torch.float64).square()
    st["w_beta"] = (2.0 / (prec @ X.square() + 1.0 / s2).sqrt()).T
    st["gam"] = gam
    st["T"] = (y @ X).T
    st["y"] = torch.tensor(d["y"], device="cuda").T
    w_nu = 0.5 / math.sqrt(gam.numel())
    st["hyp"] = torch.tensor([3.0, 0.1, *theta, *[v * v for v in sigma], 40.0 * w_nu, 0.0],
                             device="cuda", dtype=torch.float64)
    for k in ("eps", "beta"):
        st["waux_" + k] = torch.zeros_like(st[k])
    for k, v in (("eps", st["eps"]), ("beta", st["beta"]), ("gam", gam),
                 ("phi", st["hyp"][:2 * L + 2])):
        st["m_" + k] = torch.zeros_like(v)
        st["q_" + k] = torch.zeros_like(v)
    return {k: v.contiguous().clone() for k, v in st.items()}


BURNIN = 1000  # iterations before the no-allocation sweeps


def _noalloc_arrays(d, seed):
    arrays = _noalloc_state(d, seed)
    status = torch.zeros(1 + fbs.NUM_COUNTERS, dtype=torch.int64, device="cuda")
    return dict(d={k: d[k] for k in ("X", "h", "priors")}, arrays=arrays, status=status,
                it=BURNIN + 1, n_mom=0)


def _grad_inputs(L, B, seed):
    F, K = 4 * L + 1, L + L * (L + 1) // 2
    rng = np.random.default_rng(seed)
    w = [rng.normal(size=(H, F)) * math.sqrt(2.0 / F), 0.1 * rng.normal(size=H),
         rng.normal(size=(H, H)) * math.sqrt(2.0 / H), 0.1 * rng.normal(size=H),
         rng.normal(size=(K, H)) * 0.1 / math.sqrt(H), 0.05 * rng.normal(size=K)]
    return dict(params=np.concatenate([a.ravel() for a in w]).astype(np.float32),
                feat=rng.normal(size=(B, F)).astype(np.float32),
                beta=rng.normal(size=(B, L)).astype(np.float32))


# ------------------------------------------------------------------ run

def run(state):
    case, kind = state["case"], state["case"]["kind"]
    if kind == "chain":
        s = state["s"]
        s.run(case["sweeps"], burnin=state["burnin"], thin=10)
        if case["read"] == "state":
            return {**s.get_state(), **s.moments()}
        return s.estimates()
    if kind == "job":
        it = case["iters"]
        s = _sampler(state["d"], case["form"], state["seed"], trace_cap=it // 2)
        s.run(it, burnin=it // 2, thin=1)
        s.sync()
        out = s.estimates(trace_rows=it // 2)
        s.close()
        return out
    if kind == "batch":
        b = state["b"]
        b.run(case["sweeps"], burnin=TUNE, thin=10)
        # the largest outputs first; a batch of 24 gives more arrays than are
        # compared one by one, so each quantity is joined over the datasets
        est = [v.estimates() for v in b.views]
        out = {k: np.concatenate([np.ravel(e[k]) for e in est])
               for k in est[0] if k.split("_")[0] in ("mean", "sd", "lo", "hi")}
        out["evals"] = np.array([[e["counters"][k] for k in ("evals_eps", "evals_beta")]
                                 for e in est])
        if case["top"]:
            out["psi"] = b.top_level()["psi"]
        return out
    if kind == "noalloc":
        d = state["d"]
        fbs.sweep_noalloc(d["X"], d["h"], d["priors"], seed=state["seed"], it=state["it"],
                          burnin=BURNIN, n_mom=state["n_mom"], G=case["G"],
                          stream=torch.cuda.current_stream().cuda_stream,
                          status=state["status"].data_ptr(),
                          **{k: v.data_ptr() for k, v in state["arrays"].items()})
        state["it"] += 1
        state["n_mom"] += 1
        return {**{k: v for k, v in state["arrays"].items() if k not in ("y", "T")},
                "status": state["status"]}
    if kind == "train":
        s = state["s"]
        loss = s.proposal_train(epochs=1, batch=case["batch"], lr=3e-3, seed=state["seed"])
        return {"loss": loss, "params": s.proposal_params()}
    if kind == "grad":
        L = case["L"]
        loss, grad = fbs.proposal_loss_grad(state["params"], L, state["feat"], state["beta"])
        return {"loss": loss, "grad": grad}
    chains = state["chains"]
    return {"ess": [s.beta_ess() for s in chains], "rhat": fbs.rhat(chains),
            "estimates": fbs.estimates(chains)}


# ------------------------------------------------------------------ work

# Log-density evaluations of one slice update after tuning, and the operations of
# one (density, interval arithmetic) and of the update around it (random numbers,
# log-rate, moments).
EVALS, EVAL_OPS, UPDATE_OPS = 6.5, 25, 120


def _sweep_work(N, G, L, word):
    """State and counts once in, state and moments once out; the arithmetic of
    one sweep."""
    read = G * (4 * N + word * (2 * N + 2 * L + 1)) + 3 * word * G * (N + L + 1)
    write = G * word * (N + L + 1) + 2 * word * G * (N + L + 1)
    return read, write, G * (N + L) * (EVALS * EVAL_OPS + UPDATE_OPS)


def work(case):
    kind = case["kind"]
    if kind in ("chain", "job", "noalloc"):
        N, G = case["N"], case["G"]
        L = _design(case["design"], N).shape[1]
        word = 4 if case.get("form") in ("f32", "learned") else 8
        sweeps = {"chain": case.get("sweeps"), "job": case.get("iters"), "noalloc": 1}[kind]
        r, w, ops = _sweep_work(N, G, L, word)
        flops = sweeps * ops
        if case.get("form") == "learned":  # the network of every gene, every sweep
            F, K = 4 * L + 1, L + L * (L + 1) // 2
            flops += sweeps * G * 2.0 * H * (F + H + K)
        out = 8 * G * (3 * N + 3 * L + 1 + 2 * (N + L + 1)) if case.get("read") == "state" else \
            0 if kind == "noalloc" else 8 * G * 4 * (L + 1)
        return {"bytes": r + w + out, "flops": flops}
    if kind == "batch":
        total = {"bytes": 0, "flops": 0}
        for design, N, G in _batch_sizes(case):
            L = 5 if design == "paper" else 2
            r, w, ops = _sweep_work(N, G, L, 4)
            total["bytes"] += r + w + 8 * G * 4 * (L + 1)
            total["flops"] += case["sweeps"] * ops
        return total
    if kind in ("train", "grad"):
        L = case["L"] if kind == "grad" else 5
        F, K = 4 * L + 1, L + L * (L + 1) // 2
        np_ = H * (F + 1) + H * (H + 1) + K * (H + 1)
        rows = case["B"] if kind == "grad" else case["collect"] * case["G"]
        return {"bytes": 4.0 * rows * (F + L) + 16 * np_,
                "flops": rows * (6.0 * H * (F + H + K) - 2.0 * H * F)}
    G, rows, L = case["G"], case["rows"], 5
    series = 2 * G * L
    # the autocovariances of a series at the lags summed: a few tens of its rows
    return {"bytes": 8.0 * series * rows + 8 * 10 * G * L, "flops": series * rows * 2.0 * 40}


# ------------------------------------------------------------------ exact

def exact(case, seed):
    """The outputs in 64 bits by plain numpy or torch.  A chain of many sweeps in
    FP32 has no such value (its draws follow FP32 comparisons), nor has one whose
    start is itself the result of tuning sweeps; the gradient and the FP64 sweep of
    caller-owned arrays have one."""
    if case["kind"] == "grad":
        return _exact_grad(case, seed)
    if case["kind"] == "noalloc":
        return _exact_sweep(case, seed)
    return None


def _exact_grad(case, seed):
    L = case["L"]
    F, K = 4 * L + 1, L + L * (L + 1) // 2
    s = _grad_inputs(L, case["B"], seed)
    p = torch.tensor(s["params"], dtype=torch.float64, requires_grad=True)
    x, y = (torch.tensor(s[k], dtype=torch.float64) for k in ("feat", "beta"))
    sizes = [(H, F), (H,), (H, H), (H,), (K, H), (K,)]
    W1, b1, W2, b2, W3, b3 = (v.reshape(z) for v, z in zip(
        p.split([math.prod(z) for z in sizes]), sizes))
    a = torch.nn.functional.gelu(x @ W1.T + b1, approximate="tanh")
    a = torch.nn.functional.gelu(a @ W2.T + b2, approximate="tanh")
    o = a @ W3.T + b3
    C = torch.diag_embed(o[:, L:2 * L].exp())
    i, j = np.tril_indices(L, -1)
    if len(i):
        C = C.index_put((torch.arange(len(o))[:, None], torch.tensor(i), torch.tensor(j)),
                        o[:, 2 * L:])
    u = torch.linalg.solve_triangular(C, (y - o[:, :L])[:, :, None], upper=False)[:, :, 0]
    loss = (0.5 * u.square().sum(1) + o[:, L:2 * L].sum(1)).mean()
    loss.backward()
    return {"loss": float(loss.detach()), "grad": p.grad.numpy()}


# ---- one FP64 sweep in numpy (Algorithms 1 and 2 of the paper)

def _philox(index, stream, block, it, key):
    """Philox4x32-10 blocks as two 64-bit words each; index and block broadcast."""
    m = np.uint64(0xFFFFFFFF)
    index, block = np.broadcast_arrays(np.asarray(index, np.uint64), np.asarray(block, np.uint64))
    c = [index.copy(), block | np.uint64(stream << 24), np.full_like(index, it),
         np.zeros_like(index)]
    k0, k1 = key & 0xFFFFFFFF, key >> 32
    for _ in range(10):
        p0, p1 = np.uint64(0xD2511F53) * c[0], np.uint64(0xCD9E8D57) * c[2]
        c = [(p1 >> np.uint64(32)) ^ c[1] ^ np.uint64(k0), p1 & m,
             (p0 >> np.uint64(32)) ^ c[3] ^ np.uint64(k1), p0 & m]
        k0, k1 = (k0 + 0x9E3779B9) & 0xFFFFFFFF, (k1 + 0xBB67AE85) & 0xFFFFFFFF
    return c[1] << np.uint64(32) | c[0], c[3] << np.uint64(32) | c[2]


def _uniform(index, stream, k, it, key):
    k = np.asarray(k, np.uint64)
    lo, hi = _philox(index, stream, k >> np.uint64(1), it, key)
    x = np.where((k & np.uint64(1)).astype(bool), hi, lo)
    return ((x >> np.uint64(12)).astype(np.float64) + 0.5) * 2.0 ** -52


def _slice(f, x0, w, index, stream, it, key, K=100, most=100):
    """Stepping-out slice updates of many variables at once; f(i, x) is the log
    density of the variables i at x.  Returns the new values and the evaluations."""
    every = np.arange(len(x0))
    level = f(every, x0) + np.log(_uniform(index, stream, 0, it, key))
    lo = x0 - w * _uniform(index, stream, 1, it, key)
    hi = lo + w
    left = np.minimum(((K + 1) * _uniform(index, stream, 2, it, key)).astype(int), K)
    evals = len(x0)
    for end, steps, sign in ((lo, left, -1.0), (hi, K - left, 1.0)):
        i, done = every[steps > 0], 0
        while len(i):
            evals += len(i)
            i = i[level[i] < f(i, end[i])]
            end[i] += sign * w[i]
            done += 1
            i = i[steps[i] > done]
    x, i = x0.copy(), every
    for j in range(most):
        new = lo[i] + (hi[i] - lo[i]) * _uniform(index[i], stream, 3 + j, it, key)
        evals += len(i)
        ok = level[i] < f(i, new)
        x[i[ok]] = new[ok]
        i, new = i[~ok], new[~ok]
        up = new > x0[i]
        hi[i[up]], lo[i[~up]] = new[up], new[~up]
        if not len(i):
            break
    return x, evals


def _normal(index, stream, k, it, key):
    return np.sqrt(-2.0 * np.log(_uniform(index, stream, k, it, key))) * \
        np.cos(2.0 * np.pi * _uniform(index, stream, k + 1, it, key))


def _gamma(shape, index, stream, it, key):
    """Marsaglia-Tsang draws of Gamma(shape, 1), shape >= 1."""
    d = shape - 1.0 / 3.0
    c = 1.0 / math.sqrt(9.0 * d)
    out, i = np.full(len(index), float(shape)), np.arange(len(index))
    for j in range(64):
        x = _normal(index[i], stream, 4 * j, it, key)
        v = 1.0 + c * x
        u = _uniform(index[i], stream, 4 * j + 2, it, key)
        v = np.where(v > 0.0, v, np.nan) ** 3
        with np.errstate(invalid="ignore"):
            ok = (u < 1.0 - 0.0331 * x ** 4) | (np.log(u) < 0.5 * x * x + d * (1.0 - v + np.log(v)))
        ok &= ~np.isnan(v)
        out[i[ok]] = d * v[ok]
        i = i[~ok]
        if not len(i):
            break
    return out


def _exact_sweep(case, seed):
    N, G = case["N"], case["G"]
    d = _simulate(_design(case["design"], N), G, seed)
    X, h, pri = d["X"], d["h"], d["priors"]
    L = X.shape[1]
    a = {k: v.cpu().numpy() for k, v in _noalloc_state(d, seed).items()}
    it, key = BURNIN + 1, int(seed)
    y, T, hyp = a["y"], a["T"], a["hyp"]
    nu, tau, theta, sig2 = hyp[0], hyp[1], hyp[2:2 + L].copy(), hyp[2 + L:2 + 2 * L].copy()
    g = np.arange(G)
    gn = (g[None, :] * N + np.arange(N)[:, None]).ravel()
    # eps
    A = (h[:, None] + X @ a["beta"]).ravel()
    yf, hg = y.ravel().astype(float), np.tile(0.5 / a["gam"], N)

    def f_eps(i, x):
        return yf[i] * x - np.exp(A[i] + x) - x * x * hg[i]

    eps, ev_eps = _slice(f_eps, a["eps"].ravel(), a["w_eps"].ravel(), gn, 1, it, key)
    a["eps"] = eps.reshape(N, G)
    # gamma
    shape = 0.5 * (N + nu)
    a["gam"] = 0.5 * ((a["eps"] ** 2).sum(0) + nu * tau) / _gamma(shape, g, 2, it, key)
    # beta, column by column
    ev_beta = 0
    for l in range(L):
        rate = np.exp(h[:, None] + a["eps"] + X @ a["beta"])
        b0 = a["beta"][l].copy()
        values = [v for v in np.unique(X[:, l]) if v != 0.0]
        sums = [rate[X[:, l] == v].sum(0) for v in values]

        def f_beta(i, b):
            s = sum(q[i] * np.exp(v * (b - b0[i])) for v, q in zip(values, sums))
            return b * T[l][i] - s - (b - theta[l]) ** 2 * (0.5 / sig2[l])

        a["beta"][l], e = _slice(f_beta, b0, a["w_beta"][l], g * L + l, 5, it, key)
        ev_beta += e
    # hyperparameters
    S1, S2 = np.log(a["gam"]).sum(), (1.0 / a["gam"]).sum()

    def f_nu(i, v):
        x = float(v[0])
        if not 0.0 < x < pri["d"]:
            return np.array([-np.inf])
        return np.array([-G * math.lgamma(0.5 * x) + 0.5 * G * x * math.log(0.5 * x * tau) -
                         0.5 * x * (S1 + tau * S2)])

    one = np.zeros(1, int)
    nu_new, ev_nu = _slice(f_nu, np.array([nu]), np.array([hyp[2 * L + 2]]), one, 3, it, key)
    hyp[0] = nu_new[0]
    hyp[1] = _gamma(pri["a"] + 0.5 * G * hyp[0], one, 4, it, key)[0] / (pri["b"] + 0.5 * hyp[0] * S2)
    for l in range(L):
        v = 1.0 / (G / sig2[l] + 1.0 / pri["c"][l] ** 2)
        idx = np.array([l])
        th = v * a["beta"][l].sum() / sig2[l] + math.sqrt(v) * _normal(idx, 6, 0, it, key)[0]
        S = ((a["beta"][l] - th) ** 2).sum()
        s2 = 0.5 * S / _gamma(0.5 * (G - 1.0), idx, 7, it, key)[0]
        if s2 >= pri["s"][l] ** 2:  # the truncated draw went on to other attempts
            return None
        hyp[2 + l], hyp[2 + L + l] = th, s2
    for k, v in (("eps", a["eps"]), ("beta", a["beta"]), ("gam", a["gam"]),
                 ("phi", hyp[:2 * L + 2])):  # the first draw of the running moments
        a["m_" + k], a["q_" + k] = v.copy(), v * v
    return {**{k: v for k, v in a.items() if k not in ("y", "T")}, "status": None}
