"""Accepted inputs at the edges of what the kernels' shortcuts assume, and what shape AUTO's
choice by the size of the batch may not change: each against the oracle or a direct call."""
import os

import numpy as np
import pytest

from paper_1608_07058_gb300 import workloads as W
from tests.test_gpu_grid import assert_grid_parity, run_gpu_grid, run_oracle_grid
from tests.test_gpu_parity import assert_bit_parity, ml, run_gpu, run_oracle  # noqa: F401

pytestmark = pytest.mark.gpu


def torch_of(a):
    import torch
    return torch.from_numpy(np.ascontiguousarray(a)).cuda()


@pytest.mark.parametrize("d", [2**32 - 2, 2**32 - 1, 2**32, 2**33 + 5, 2**62])
@pytest.mark.parametrize("bins", [1, 2, 3, 4096])
def test_kl_ranges_around_32_bits(ml, oracle, d, bins):
    """Pooled ranges around 2^32, where the range fits 32 bits and the width of one bin does
    not: every value has a bin below max_bins."""
    rng = np.random.default_rng(3)
    lo = -(d // 2)
    a = np.array([lo, lo + d] + [lo + int(u * d) for u in rng.random(398)], np.int64)
    b = np.array([lo + int(u * u * d) for u in rng.random(300)], np.int64)
    kl, mean = ml.ml_kl_divergence(torch_of(a.reshape(-1, 1, 1)), torch_of(b.reshape(-1, 1, 1)),
                                   bins)
    want, want_mean = oracle.kl_grid(a.reshape(-1, 1, 1), b.reshape(-1, 1, 1), bins)
    assert np.array_equal(kl.cpu().numpy(), np.asarray(want).reshape(1, 1))
    assert float(mean) == float(want_mean)


@pytest.mark.parametrize("mode", [0, 2])
@pytest.mark.parametrize("kw", [dict(shape=1), dict(shape=2), dict(shape=4), dict(shape=6, form=1),
                                dict(shape=1, specialize=1), dict(shape=6, form=1, specialize=1)])
def test_infinite_rate_of_an_absent_reactant(ml, oracle, mode, kw):
    """theta = +inf is accepted (not negative, not NaN); with g = 0 the propensity and a0 are
    NaN.  An SSA firing's time is then NaN: it is not past T, fires, and ends the trajectory
    after its burst, in every driver as in the oracle."""
    crn = W._crn("absent", 2, [({0: 1}, {}, 1.0), ({}, {1: 1}, 5.0), ({1: 1}, {}, 1.0)])
    n = 70
    theta = np.tile([np.inf, 5.0, 1.0], (n, 1))
    T = np.linspace(0.1, 2.0, n)
    args = dict(theta=theta, seed=21, mode=mode, max_steps=50)
    o = run_oracle(oracle, crn, n, [0, 10], T, **args)
    if mode == 2:
        assert np.isnan(o["G"]).all() and (o["counters"][:, 2] == 100).all()
    g = run_gpu(ml, crn, n, [0, 10], T, **args, **kw)
    for key in ("X", "r", "status", "counters"):
        assert np.array_equal(g[key], o[key]), key
    assert np.array_equal(g["G"], o["G"], equal_nan=True)
    if mode == 2:  # fast precision: the same firings
        f = run_gpu(ml, crn, n, [0, 10], T, precision=ml.ML_PREC_FAST_FP32, **args, **kw)
        for key in ("X", "r", "status", "counters"):
            assert np.array_equal(f[key], o[key]), key
        assert np.isnan(f["G"]).all()


@pytest.mark.parametrize("first,then", [(100, 6000), (6000, 100)])
@pytest.mark.parametrize("specialize", [0, 1])
@pytest.mark.parametrize("grid", [False, True])
def test_warm_up_of_any_size_covers_a_captured_call(ml, first, then, specialize, grid):
    """Shape AUTO takes another kernel for another size of the batch: a call captured after
    one warm-up of a size on the other side of the line allocates and loads nothing."""
    import torch
    crn = W.dimerisation()
    x0 = torch.tensor([400, 798, 0], device="cuda")
    T = torch.full((1,), 0.02, dtype=torch.float64, device="cuda")
    t_obs = torch.tensor([0.01, 0.02], dtype=torch.float64, device="cuda")
    params = ml.ml_default_params(form=ml.ML_FORM_PERSISTENT, specialize=specialize)

    def call(model, n):
        if grid:
            return ml.ml_simulate_grid(model, n, x0, T, t_obs, params=params, seed=5)
        return ml.ml_simulate(model, n, x0, T, params=params, seed=5)

    model = ml.model_from_crn(crn)
    call(model, first)
    torch.cuda.synchronize()
    graph = torch.cuda.CUDAGraph()
    with torch.cuda.graph(graph):
        out = call(model, then)
    graph.replay()
    torch.cuda.synchronize()
    want = call(ml.model_from_crn(crn), then)
    torch.cuda.synchronize()
    for key in want:
        assert torch.equal(out[key], want[key]), key


def test_posterior_huge_shapes(ml, oracle):
    """Shapes on both sides of the FP32 estimate's range and far beyond it, where the FP64
    acceptance test is its own rounding noise: every draw is the oracle's."""
    alpha = np.array([6.8e10, 6.9e10, 1e12, 1e13, 1e14, 1e15, 1e17, 1e300])
    n, M = 4000, alpha.size
    beta, r, G = np.ones(M), np.zeros((n, M), np.int64), np.zeros((n, M))
    th, st = ml.ml_posterior_sample(*(torch_of(a) for a in (alpha, beta, r, G)), seed=17)
    want, want_st = oracle.posterior_sample(alpha, beta, r, G, seed=17, traj_id_base=0)
    differ = (th.cpu().numpy() != want).sum(0)
    assert not differ.any(), dict(zip(alpha, differ))
    assert np.array_equal(st.cpu().numpy().astype(np.uint32), want_st)


def test_reciprocals_of_the_fast_newton_system(tmp_path):
    """Before its last rounding the reciprocal is within 2^-63 (the third power of FP32's
    2^-21), so it may differ from the division's only where 1/b lies within 2^-10 ulp of a
    midpoint: at most 2^-9 of the values, by one unit in the last place."""
    import subprocess
    from paper_1608_07058_gb300 import build as B
    exe = str(tmp_path / "recip_check")
    src = os.path.join(os.path.dirname(os.path.abspath(__file__)), "recip_check.cu")
    cmd = [B._nvcc(), *B.ARCH, "-O2", "-std=c++17", "-I", B.CSRC, "-I", B.INCLUDE, src, "-o", exe]
    assert subprocess.run(cmd, capture_output=True, text=True).returncode == 0
    res = subprocess.run([exe], capture_output=True, text=True, timeout=120)
    assert res.returncode == 0
    n, differ, ulps = map(int, res.stdout.split())
    assert n == 2**24 and differ <= n * 2**-9 and ulps <= 1


# Reference precision with the shape named, so that both kernels run whatever shape AUTO would
# choose for these sizes: (shape, compiled for the model).
KERNELS = [(1, 0), (1, 1), (2, 0)]


@pytest.mark.parametrize("shape,specialize", KERNELS)
@pytest.mark.parametrize("form", [0, 1])
@pytest.mark.parametrize("n", [1, 31, 33, 257, 607, 609])
def test_reference_tiny_batches_per_shape(ml, oracle, shape, specialize, form, n):
    """Around a warp and around the batch that is spread one trajectory to a warp (608 on 152
    SMs), per-trajectory rate constants and horizons (some zero)."""
    crn = W.gene_expression()
    rng = np.random.default_rng(n)
    theta = rng.gamma(2.0, crn.rates / 2.0, size=(n, 6))
    T = rng.uniform(0.0, 6.0, n)
    T[::7] = 0.0
    g = run_gpu(ml, crn, n, [1, 2, 20], T, theta, seed=8, shape=shape, specialize=specialize,
                form=form)
    o = run_oracle(oracle, crn, n, [1, 2, 20], T, theta, seed=8)
    assert_bit_parity(g, o, f"n={n}")


@pytest.mark.parametrize("shape,specialize", KERNELS)
def test_reference_inputs_per_trajectory_per_shape(ml, oracle, shape, specialize):
    """Per-trajectory x0, T and theta with an id offset, and the gene-expression batch."""
    kw = dict(shape=shape, specialize=specialize)
    w = W.config(1, n_traj=700)
    rng = np.random.default_rng(2)
    x0 = rng.integers(0, 500, size=(700, 3))
    T = rng.uniform(0.0, 0.3, size=700)
    T[:5] = 0.0
    theta = np.abs(w.crn.rates * rng.gamma(2.0, 0.5, size=(700, 4)))
    args = dict(seed=2**40 + 9, base=123456)
    assert_bit_parity(run_gpu(ml, w.crn, 700, x0, T, theta, **args, **kw),
                      run_oracle(oracle, w.crn, 700, x0, T, theta, **args), "per-trajectory")
    w = W.config(2, n_traj=400)
    assert_bit_parity(run_gpu(ml, w.crn, 400, w.x0, w.T, w.theta, seed=3, **kw),
                      run_oracle(oracle, w.crn, 400, w.x0, w.T, w.theta, seed=3), "gene")


@pytest.mark.parametrize("shape", [1, 2])
def test_reference_forms_per_shape(ml, shape):
    """Plain, persistent, graph and host calls of one shape give the same results."""
    w = W.config(2, n_traj=1500)
    T = w.T * 0.2
    model = ml.model_from_crn(w.crn)
    calls = [dict(), dict(form=1, block_size=64, ctas_per_sm=2), dict(form=1, use_graph=1)]
    if shape == 1:
        calls += [dict(specialize=1), dict(form=1, use_graph=1, specialize=1)]
    runs = [run_gpu(ml, w.crn, w.n_traj, w.x0, T, w.theta, seed=4, model=model, shape=shape, **kw)
            for kw in calls]
    host = ml.ml_simulate_host(model, w.n_traj, w.x0, T, w.theta,
                               params=ml.ml_default_params(shape=shape, max_steps=200_000), seed=4)
    host["status"] = host["status"].astype(np.uint32)
    for other in runs[1:] + [host]:
        for key in runs[0]:
            assert np.array_equal(runs[0][key], other[key]), key


@pytest.mark.parametrize("shape", [1, 2])
def test_reference_time_grid_per_shape(ml, oracle, shape):
    """Per-trajectory horizons below, at and above grid points, and gene expression."""
    rng = np.random.default_rng(4)
    for crn, x0, T, grid in ((W.dimerisation(), [400, 798, 0], rng.uniform(0.01, 0.3, 1000),
                              [0.0, 0.05, 0.1, 0.2, 0.25]),
                             (W.gene_expression(), [1, 2, 20], rng.uniform(1.0, 20.0, 300),
                              [0.5, 5.0, 5.0, 12.0])):
        g = run_gpu_grid(ml, crn, T.size, x0, T, grid, seed=2, shape=shape)
        o = run_oracle_grid(oracle, crn, T.size, x0, T, grid, seed=2)
        assert_grid_parity(g, o, crn.name)
