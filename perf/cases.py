"""The work that users of this framework have it do, as cases that can be timed: simulate
calls of the four networks of `workloads.py` in both precisions and both launch forms, the
host-buffer call, time-grid output, the accuracy metric and the Bayesian step.

A case is a dict of plain values.  `listed` gives the standing cases, `draw` another one of
the same ranges, `prepare` what a program holds before the call, `run` one pass through the
public entry points, `work` the bytes and operations that pass cannot do without, `exact`
its floating-point results in plain numpy where they have a closed definition.
"""
import functools
import math

import numpy as np
import torch

from paper_1608_07058_gb300 import matleap as ml
from paper_1608_07058_gb300 import workloads as W

CONFIG = {"immigration_death": 0, "dimerisation": 1, "gene_expression": 2, "random_50x100": 3}


def _sim(name, net, n, precision, form, horizon, spread=0.0, ragged=False, specialize=False,
         shape="auto", graph=False, path="device", points=0, jacobian="fd", mode="adaptive"):
    """horizon: T, or the largest T where it is ragged (T x U[0.5, 1] per trajectory, the
    gene-expression batch U[0.25, 1]); spread: shape of the per-trajectory Gamma rate
    constants around the model's (0: the model's own); points: time-grid points."""
    return {"name": name, "path": path, "net": net, "n": n, "precision": precision,
            "form": form, "horizon": horizon, "spread": spread, "ragged": ragged,
            "specialize": specialize, "shape": shape, "graph": graph, "points": points,
            "jacobian": jacobian, "mode": mode}


def listed():
    return [
        # The smallest calls: a user tries a model out with the default parameters
        # (reference precision, one plain launch).  One serial chain of firings per thread.
        _sim("immigration_ref_100", "immigration_death", 100, "ref", "plain", 100.0),
        # The first benchmark configuration in the fast form: short serial chains, a batch
        # that fills a fraction of the GPU, no kernels compiled for the model.
        _sim("immigration_fast_10k", "immigration_death", 10_000, "fast", "persistent", 100.0),
        # The paper's stiff third model with the default parameters, as a first script runs
        # it: implicit leaps in reference precision.
        _sim("dimerisation_ref_100k", "dimerisation", 100_000, "ref", "plain", 0.2),
        # The same batch with the parameters that the README recommends.
        _sim("dimerisation_fast_100k", "dimerisation", 100_000, "fast", "persistent", 0.2,
             specialize=True),
        # The benchmark's headline: a particle filter's whole batch, every particle with its
        # own rate constants and horizon (bursts of exact SSA between explicit leaps).
        _sim("gene_fast_1m", "gene_expression", 1_000_000, "fast", "persistent", 200.0, 2.0,
             True, specialize=True, shape="pool", graph=True),
        # A validation run of the same filter in reference precision, an odd batch.
        _sim("gene_ref_10k", "gene_expression", 10_007, "ref", "persistent", 200.0, 2.0, True),
        # A service's request: numpy or pinned host buffers in and out, per-trajectory rate
        # constants and the serving mix's short horizons, precompiled kernels.
        _sim("gene_host_30k", "gene_expression", 30_011, "fast", "persistent", 6.0, 2.0, True,
             graph=True, path="host"),
        # The large network, one trajectory per warp: bursts of SSA between implicit leaps
        # (a 50 x 50 Newton system each).  The benchmark's T = 10 is 200 times this.
        _sim("random_crn_fast_4k", "random_50x100", 4_096, "fast", "persistent", 0.05),
        # The serving mix's requests of the large network, in reference precision: short
        # horizons, spread rate constants, SSA bursts only.
        _sim("random_crn_ref_1500", "random_50x100", 1_500, "ref", "plain", 5e-4, 2.0, True),
        # The accuracy study: 10,000 trajectories observed at 20 points (a leap ends at each).
        _sim("grid_dimerisation_10k", "dimerisation", 10_000, "fast", "persistent", 0.2,
             path="grid", points=20),
        # The accuracy study's metric on two such samples.
        {"name": "kl_10k", "path": "kl", "n_ref": 10_000, "n_test": 10_000, "points": 20,
         "species": 3, "max_bins": 1024},
        # The Bayesian step after the headline batch: a posterior draw of every rate
        # constant, then systematic resampling by the particles' weights.
        {"name": "bayes_1m", "path": "bayes", "n": 1_000_000, "reactions": 6},
    ]


def _log_int(rng, lo, hi):
    return min(hi, max(lo, int(round(math.exp(rng.uniform(math.log(lo), math.log(hi)))))))


def draw(rng):
    """One more case: path, network, sizes (spread over their logarithm), precision, form and
    options as users combine them."""
    kind = rng.choice(["immigration", "dimerisation", "gene", "gene", "crn", "host", "grid",
                       "kl", "bayes"])
    fast = rng.random() < 0.6
    precision = "fast" if fast else "ref"
    form = "persistent" if fast or rng.random() < 0.4 else "plain"
    specialize = form == "persistent" and rng.random() < 0.5
    shape = rng.choice(["auto", "auto", "pool", "seq"]) if form == "persistent" else "auto"
    graph = form == "persistent" and rng.random() < 0.3
    jac = rng.choice(["fd", "fd", "analytic"])
    if kind == "kl":
        c = {"path": "kl", "n_ref": _log_int(rng, 500, 20_000), "n_test": _log_int(rng, 500, 20_000),
             "points": rng.randint(3, 50), "species": rng.randint(1, 4),
             "max_bins": rng.choice([100, 1024, 4096])}
    elif kind == "bayes":
        c = {"path": "bayes", "n": _log_int(rng, 300, 1_000_000), "reactions": rng.choice([2, 4, 6])}
    elif kind == "immigration":
        c = _sim("", "immigration_death", _log_int(rng, 50, 30_000), precision, form,
                 rng.uniform(20.0, 100.0), rng.choice([0.0, 2.0]), rng.random() < 0.5,
                 specialize, shape, graph)
    elif kind == "dimerisation":
        c = _sim("", "dimerisation", _log_int(rng, 100, 100_000), precision, form,
                 rng.uniform(0.05, 0.2), rng.choice([0.0, 50.0]), rng.random() < 0.5,
                 specialize, shape, graph, jacobian=jac)
    elif kind == "gene":
        n = _log_int(rng, 500, 400_000 if fast else 8_000)
        c = _sim("", "gene_expression", n, precision, form, rng.uniform(50.0, 200.0), 2.0, True,
                 specialize, shape, graph)
    elif kind == "host":
        net, T, k = rng.choice([("immigration_death", 50.0, 2.0), ("dimerisation", 0.2, 50.0),
                                ("gene_expression", 6.0, 2.0)])
        c = _sim("", net, _log_int(rng, 1_000, 100_000), "fast", "persistent", T, k, True,
                 specialize, "auto", graph, path="host")
    elif kind == "grid":
        net, T, k = rng.choice([("dimerisation", 0.2, 0.0), ("immigration_death", 50.0, 0.0),
                                ("gene_expression", 20.0, 2.0)])
        c = _sim("", net, _log_int(rng, 500, 20_000), precision, form, T, k, False,
                 path="grid", points=rng.randint(3, 50), jacobian=jac)
    elif rng.random() < 0.5:  # the large network, as the serving mix asks for it
        c = _sim("", "random_50x100", _log_int(rng, 100, 10_000), precision, form,
                 rng.uniform(2e-4, 5e-4), 2.0, True)
    else:  # the large network over a longer horizon, with its implicit leaps
        c = _sim("", "random_50x100", _log_int(rng, 100, 4_096 if fast else 1_024), precision,
                 form, rng.uniform(0.005, 0.05 if fast else 0.02), jacobian=jac)
    c.pop("name", None)
    return c


@functools.lru_cache(maxsize=None)
def _network(net):
    """(reaction network, initial state) of a benchmark configuration."""
    w = W.config(CONFIG[net], n_traj=1)
    return w.crn, w.x0


@functools.lru_cache(maxsize=None)
def _model(net):
    """The model handle: a program creates it once and keeps it for all its calls."""
    return ml.model_from_crn(_network(net)[0])


SHAPES = {"auto": ml.ML_SHAPE_AUTO, "pool": ml.ML_SHAPE_THREAD_POOL, "seq": ml.ML_SHAPE_THREAD_SEQ}


def _params(case):
    if case["precision"] == "ref" and case["form"] == "plain" and case["jacobian"] == "fd":
        return None  # the defaults
    fast = case["precision"] == "fast"
    return ml.ml_default_params(
        precision=ml.ML_PREC_FAST_FP32 if fast else ml.ML_PREC_REF_FP64,
        form=ml.ML_FORM_PERSISTENT if case["form"] == "persistent" else ml.ML_FORM_PLAIN,
        shape=SHAPES[case["shape"]], specialize=int(case["specialize"]),
        use_graph=int(case["graph"]),
        jacobian=ml.ML_JAC_ANALYTIC if case["jacobian"] == "analytic" else ml.ML_JAC_FD)


def _bayes_inputs(case, seed):
    """Prior, firing counts and integrals as the gene-expression batch leaves them (counts
    from none to thousands, skewed by the particles' own rate constants), and log-weights."""
    n, M = case["n"], case["reactions"]
    rng = np.random.default_rng(seed)
    rate = np.array(W.GENE_THETA_TRUE[:M])
    alpha, beta = np.full(M, 2.0), 2.0 / rate
    G = rng.gamma(2.0, 40.0, size=(n, M))
    G[rng.random((n, M)) < 0.02] = 0.0  # a gene that never switched on
    r = rng.poisson(rng.gamma(2.0, rate / 2.0, size=(n, M)) * G).astype(np.int64)
    logw = -0.5 * rng.chisquare(3.0, size=n) * rng.choice([1.0, 4.0], size=n)
    return alpha, beta, r, G, logw


def _kl_inputs(case, seed):
    """Two samples of counts over time: the first species spread over hundreds of counts, the
    others over tens, the test sample narrower, as leaping leaves it."""
    rng = np.random.default_rng(seed)
    K, N = case["points"], case["species"]
    mean = rng.uniform(20.0, 6000.0, size=(K, N))
    sd = np.sqrt(mean)
    ref = rng.normal(mean, sd, size=(case["n_ref"], K, N))
    test = rng.normal(mean, 0.6 * sd, size=(case["n_test"], K, N))
    return (np.maximum(np.rint(ref), 0).astype(np.int64),
            np.maximum(np.rint(test), 0).astype(np.int64))


def prepare(case, seed):
    dev = torch.device("cuda")
    if case["path"] == "bayes":
        alpha, beta, r, G, logw = _bayes_inputs(case, seed)
        return {"case": case, "seed": seed + 1,
                "in": [torch.from_numpy(a).to(dev) for a in (alpha, beta, r, G)],
                "logw": torch.from_numpy(logw).to(dev),
                "ws": torch.empty(ml.ml_resample_workspace_bytes(case["n"]), dtype=torch.uint8,
                                  device=dev)}
    if case["path"] == "kl":
        ref, test = _kl_inputs(case, seed)
        return {"case": case, "ref": torch.from_numpy(ref).to(dev),
                "test": torch.from_numpy(test).to(dev)}
    crn, x0 = _network(case["net"])
    n, rng = case["n"], np.random.default_rng(seed)
    theta = None
    if case["spread"]:
        theta = rng.gamma(case["spread"], crn.rates / case["spread"], size=(n, crn.n_reactions))
    if case["ragged"]:
        low = 0.25 if case["net"] == "gene_expression" and case["path"] == "device" else 0.5
        T = case["horizon"] * rng.uniform(low, 1.0, size=n)
    else:
        T = np.array([case["horizon"]])
    state = {"case": case, "model": _model(case["net"]), "params": _params(case),
             "seed": seed + 1}
    x0, T = torch.from_numpy(x0.copy()), torch.from_numpy(T)
    theta = None if theta is None else torch.from_numpy(theta)
    if case["path"] == "host":
        pin = lambda *s: torch.empty(s, dtype=torch.int64, pin_memory=True)  # noqa: E731
        state["x0"], state["T"], state["theta"] = (
            None if a is None else a.pin_memory() for a in (x0, T, theta))
        N, M = crn.n_species, crn.n_reactions
        state["out"] = {"X": pin(n, N), "r": pin(n, M), "G": pin(n, M).view(torch.float64),
                        "status": torch.empty(n, dtype=torch.int32, pin_memory=True),
                        "counters": pin(n, 4)}
        return state
    state["x0"], state["T"], state["theta"] = (
        None if a is None else a.to(dev) for a in (x0, T, theta))
    if case["points"]:
        K = case["points"]
        state["t_obs"] = torch.linspace(case["horizon"] / K, case["horizon"], K,
                                        dtype=torch.float64, device=dev)
    return state


def run(state):
    case = state["case"]
    if case["path"] == "bayes":
        theta, status = ml.ml_posterior_sample(*state["in"], seed=state["seed"])
        ancestors = ml.ml_resample_systematic(state["logw"], seed=state["seed"],
                                              workspace=state["ws"])
        return {"theta": theta, "status": status, "ancestors": ancestors}
    if case["path"] == "kl":
        kl, mean = ml.ml_kl_divergence(state["ref"], state["test"], max_bins=case["max_bins"])
        return {"kl": kl, "mean": mean}
    args = (state["model"], case["n"], state["x0"], state["T"])
    if case["path"] == "host":
        return ml.ml_simulate_host(*args, theta=state["theta"], params=state["params"],
                                   seed=state["seed"], out=state["out"])
    if case["points"]:
        return ml.ml_simulate_grid(*args, state["t_obs"], theta=state["theta"],
                                   params=state["params"], seed=state["seed"])
    return ml.ml_simulate(*args, theta=state["theta"], params=state["params"],
                          seed=state["seed"])


# Mean events of one trajectory, counted with the CPU reference: (explicit leaps, implicit
# leaps, SSA firings) over the horizon named.  They grow in proportion to the horizon; a
# time grid adds a leap per point.  Gene expression's horizons average 0.625 T.
EVENTS = {"immigration_death": (100.0, 20.6, 0.0, 1667.0), "dimerisation": (0.2, 0.0, 14.0, 1.0),
          "gene_expression": (125.0, 443.0, 0.0, 5321.0), "random_50x100": (0.05, 0.0, 24.0, 12300.0)}
RANDOM_OPS = 76  # ten Philox rounds of seven integer operations, and two uniforms
NEWTON_ITERATIONS = 4.3


def _event_ops(crn):
    """Arithmetic of an explicit leap, an implicit leap and an SSA firing of a network."""
    N, M = crn.n_species, crn.n_reactions
    props = int(2 * (crn.orders > 0).sum() + M)
    nnz = int((crn.stoich != 0).sum())
    ssa = props + 4 * M + RANDOM_OPS + 20 + 2 * nnz / M
    leap = 2 * props + 4 * M + 5 * nnz + 7 * N + M * (RANDOM_OPS + 40)
    newton = props + 6 * nnz + 2 * N ** 3 / 3 + 2 * N * N + 7 * N
    return leap, leap + NEWTON_ITERATIONS * newton, ssa


def work(case):
    if case["path"] == "bayes":
        n, M = case["n"], case["reactions"]
        # per draw r and G in, theta out, two random blocks, three logarithms, a square root
        # and two divisions; per particle a log-weight in, an ancestor out, an exponential
        return {"bytes": n * (24 * M + 4) + 16 * n + 16 * M, "flops": n * (260 * M + 40)}
    if case["path"] == "kl":
        KN = case["points"] * case["species"]
        return {"bytes": 8 * KN * (case["n_ref"] + case["n_test"] + 1) + 8,
                "flops": KN * (4 * (case["n_ref"] + case["n_test"]) + 100 * 300)}
    crn, _ = _network(case["net"])
    n, N, M, K = case["n"], crn.n_species, crn.n_reactions, case["points"]
    T0, ex, im, ssa = EVENTS[case["net"]]
    low = 0.25 if case["net"] == "gene_expression" and case["path"] == "device" else 0.5
    share = case["horizon"] / T0 * ((1.0 + low) / 2.0 if case["ragged"] else 1.0)
    leap_ops, implicit_ops, ssa_ops = _event_ops(crn)
    flops = n * (share * (ex * leap_ops + im * implicit_ops + ssa * ssa_ops) + K * leap_ops)
    nbytes = n * (8 * N + 16 * M + 4 + 32 + 8 * N * K) + 8 * N + 8 * K
    nbytes += n * 8 * M if case["spread"] else 8 * M
    nbytes += 8 * (n if case["ragged"] else 1)
    return {"bytes": float(nbytes), "flops": float(flops)}


# ---- plain numpy of what has a closed definition -----------------------------------------

def _philox(seed, c0, c1, c3):
    """Words of Philox4x32-10 with key `seed` at counters (c0, c1, 0, c3), as uint64."""
    m32 = np.uint64(0xFFFFFFFF)
    c = [np.asarray(c0, np.uint64), np.asarray(c1, np.uint64),
         np.zeros(np.shape(c0), np.uint64), np.asarray(c3, np.uint64)]
    k0, k1 = seed & 0xFFFFFFFF, (seed >> 32) & 0xFFFFFFFF
    for _ in range(10):
        a, b = np.uint64(0xD2511F53) * c[0], np.uint64(0xCD9E8D57) * c[2]
        c = [(b >> np.uint64(32)) ^ c[1] ^ np.uint64(k0), b & m32,
             (a >> np.uint64(32)) ^ c[3] ^ np.uint64(k1), a & m32]
        k0, k1 = (k0 + 0x9E3779B9) & 0xFFFFFFFF, (k1 + 0xBB67AE85) & 0xFFFFFFFF
    return c


def _uniform(hi, lo):
    n = (hi >> np.uint64(6)).astype(np.float64) * 2.0 ** 26 + (lo >> np.uint64(6)).astype(np.float64)
    return (n + 0.5) * 2.0 ** -52


def _gamma_draws(shape, rate, seed, ids, stream):
    """Gamma(shape, rate) by Marsaglia & Tsang (2000) on the counters of the posterior draw;
    NaN where shape or rate is not positive."""
    out = np.full(shape.shape, np.nan)
    todo = np.flatnonzero((shape > 0) & (rate > 0))
    for t in range(64):
        if not todo.size:
            break
        a = np.where(shape[todo] < 1.0, shape[todo] + 1.0, shape[todo])
        d = a - 1.0 / 3.0
        c1 = np.uint64(0x80000000) + stream[todo]
        w = _philox(seed, ids[todo], c1, np.full(todo.size, 2 * t))
        v1, v2 = 2.0 * _uniform(w[0], w[1]) - 1.0, 2.0 * _uniform(w[2], w[3]) - 1.0
        s = v1 * v1 + v2 * v2
        w = _philox(seed, ids[todo], c1, np.full(todo.size, 2 * t + 1))
        u, ub = _uniform(w[0], w[1]), _uniform(w[2], w[3])
        with np.errstate(all="ignore"):
            z = v1 * np.sqrt(-2.0 * np.log(s) / s)
            v = (1.0 + z / np.sqrt(9.0 * d)) ** 3
            ok = (s < 1.0) & (s > 0.0) & (v > 0.0)
            ok &= np.log(u) < 0.5 * z * z + d - d * v + d * np.log(v)
            x = d * v * np.where(shape[todo] < 1.0, ub ** (1.0 / shape[todo]), 1.0)
        out[todo[ok]] = x[ok] / rate[todo[ok]]
        todo = todo[~ok]
    return out


def exact(case, seed):
    if case["path"] == "bayes":
        alpha, beta, r, G, _ = _bayes_inputs(case, seed)
        n, M = r.shape
        ids = np.repeat(np.arange(n, dtype=np.uint64), M)
        theta = _gamma_draws((alpha + r).ravel(), (beta + G).ravel(), seed + 1, ids,
                             np.tile(np.arange(M, dtype=np.uint64), n))
        return {"theta": theta.reshape(n, M), "status": None, "ancestors": None}
    if case["path"] == "kl":
        ref, test = _kl_inputs(case, seed)
        K, N = case["points"], case["species"]
        kl = np.empty((K, N))
        for k in range(K):
            for s in range(N):
                a, b = ref[:, k, s], test[:, k, s]
                lo, hi = min(a.min(), b.min()), max(a.max(), b.max())
                w = (hi - lo) // case["max_bins"] + 1
                bins = int((hi - lo) // w + 1)
                p = np.bincount((a - lo) // w, minlength=bins) + 0.5
                q = np.bincount((b - lo) // w, minlength=bins) + 0.5
                p, q = p / p.sum(), q / q.sum()
                kl[k, s] = float((p * np.log(p / q)).sum())
        return {"kl": kl, "mean": np.array([kl.mean()])}
    return None  # a simulation's results are those of its random choices, step by step
