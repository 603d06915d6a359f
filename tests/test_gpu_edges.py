"""Accepted inputs at the edges of what the kernels' shortcuts assume, and what shape AUTO's
choice by the size of the batch may not change: each against the oracle or a direct call."""
import os

import numpy as np
import pytest

from paper_1608_07058_gb300 import workloads as W
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
