"""Where a call's kernel is chosen by its size, and where values change their form: both
sides of each line give the same results.

Reference precision is compared with the oracle bit for bit.  Fast precision is keyed by
trajectory id, so a batch spread thinly over the warps equals the same ids of a batch that
fills them, exactly.
"""
import numpy as np
import pytest

from paper_1608_07058_gb300 import workloads as W
from tests.test_gpu_parity import assert_bit_parity, ml, run_gpu, run_oracle  # noqa: F401

pytestmark = pytest.mark.gpu


def _inputs(net, n, seed=5):
    crn = {"id": W.immigration_death, "dim": W.dimerisation, "gene": W.gene_expression}[net]()
    rng = np.random.default_rng(seed)
    k = 50.0 if net == "dim" else 2.0
    theta = rng.gamma(k, crn.rates / k, size=(n, crn.n_reactions))
    T = {"id": 2.0, "dim": 0.02, "gene": 4.0}[net] * rng.uniform(0.5, 1.0, size=n)
    x0 = {"id": [3], "dim": [400, 798, 0], "gene": [1, 2, 20]}[net]
    return crn, theta, T, x0


@pytest.mark.parametrize("net,n", [("id", 1216), ("id", 1217), ("dim", 4864), ("dim", 4865),
                                   ("gene", 1), ("gene", 14592), ("gene", 14593)])
@pytest.mark.parametrize("ragged", [False, True])
def test_reference_shape_auto_equals_both_kernels(ml, net, n, ragged):
    crn, theta, T, x0 = _inputs(net, n)
    args = dict(theta=theta if ragged else None, seed=3, form=ml.ML_FORM_PERSISTENT)
    Tn = T if ragged else T[:1]
    auto = run_gpu(ml, crn, n, x0, Tn, **args)
    for shape in (ml.ML_SHAPE_THREAD, ml.ML_SHAPE_WARP):
        other = run_gpu(ml, crn, n, x0, Tn, shape=shape, **args)
        for key in auto:
            assert np.array_equal(auto[key], other[key]), (shape, key)


@pytest.mark.parametrize("shape", ["ML_SHAPE_THREAD", "ML_SHAPE_THREAD_SEQ", "ML_SHAPE_THREAD_POOL"])
@pytest.mark.parametrize("n", [1, 31, 33, 607, 609, 5000])
@pytest.mark.parametrize("specialize", [0, 1])
def test_fast_results_do_not_depend_on_the_spread(ml, shape, n, specialize):
    crn, theta, T, x0 = _inputs("gene", 25_000)
    model = ml.model_from_crn(crn)
    args = dict(seed=9, model=model, precision=ml.ML_PREC_FAST_FP32,
                form=ml.ML_FORM_PERSISTENT, shape=getattr(ml, shape), specialize=specialize)
    full = run_gpu(ml, crn, 25_000, x0, T, theta, **args)
    part = run_gpu(ml, crn, n, x0, T[:n], theta[:n], **args)
    for key in part:
        assert np.array_equal(part[key], full[key][:n]), key


@pytest.mark.parametrize("count", [2**24 + 1, 2**31 - 1, 2**32 + 3, 2**47 + 1, 2**53 + 3, 2**60])
@pytest.mark.parametrize("shape", ["ML_SHAPE_THREAD", "ML_SHAPE_WARP"])
def test_reference_counts_across_the_conversions(ml, oracle, count, shape):
    """Counts around the edges of the integer forms of the conversions, the second-order
    count whose C(x, 2) leaves them, and Poisson means on both sides of the PTRS estimate's
    range.  Rates keep the leaps' means below 2^48."""
    rate = min(1.0, 2.0**40 / count)
    for crn, x0 in ((W.isomerisation(rate, 2.0 * rate), [count, count // 2]),
                    (W.dimerisation((rate, rate * 1e-6 / count, 1e-3 * rate, rate)), [count, 7, 0])):
        args = dict(seed=11, max_steps=60)
        g = run_gpu(ml, crn, 64, x0, 1.0, shape=getattr(ml, shape), **args)
        o = run_oracle(oracle, crn, 64, x0, 1.0, **args)
        assert_bit_parity(g, o, f"{crn.name} {count}")


@pytest.mark.parametrize("mean", [0.5, 9.99, 10.01, 30.0, 1e3, 3e5, 9.9e8, 1.1e9])
@pytest.mark.parametrize("shape", ["ML_SHAPE_THREAD", "ML_SHAPE_WARP"])
def test_reference_poisson_estimates_decide_as_the_oracle(ml, oracle, mean, shape):
    """A source-only network leaps once to T, so X(T) is one Poisson draw: 20,000 of them at
    means on both sides of inversion and PTRS and of the estimates' range."""
    crn = W._crn("source", 1, [({}, {0: 1}, mean)])
    args = dict(seed=13, ssa_factor=0.0)
    g = run_gpu(ml, crn, 20_000, [0], 1.0, shape=getattr(ml, shape), **args)
    o = run_oracle(oracle, crn, 20_000, [0], 1.0, **args)
    assert_bit_parity(g, o, f"mean {mean}")


@pytest.mark.parametrize("n_ref,n_test,spread,bins", [(1, 1, 0, 1024), (700, 1, 3000, 4096),
                                                      (9000, 8192, 300, 1024), (8193, 33, 40, 7),
                                                      (20000, 20000, 2, 1024), (5000, 64, 2**40, 4096)])
def test_kl_tables_and_batches(ml, oracle, n_ref, n_test, spread, bins):
    """Samples around the load batch, counts above and below the table, one bin and 4,096."""
    import torch
    rng = np.random.default_rng(n_ref)
    a = rng.integers(-spread, spread + 1, size=(n_ref, 2, 2))
    b = rng.integers(-spread // 2, spread // 2 + 1, size=(n_test, 2, 2))
    kl, mean = ml.ml_kl_divergence(torch.from_numpy(a).cuda(), torch.from_numpy(b).cuda(), bins)
    want, want_mean = oracle.kl_grid(a, b, bins)
    assert np.array_equal(kl.cpu().numpy(), np.asarray(want).reshape(2, 2))
    assert float(mean) == float(want_mean)


@pytest.mark.parametrize("order", ["random", "increasing", "equal", "one", "ninf"])
@pytest.mark.parametrize("n", [1, 1023, 1024, 1025, 49_153, 200_001])
def test_resampling_block_edges(ml, oracle, n, order):
    import torch
    rng = np.random.default_rng(n)
    logw = {"random": rng.normal(0, 5, n), "increasing": np.linspace(-40, 0, n), "equal": np.zeros(n),
            "one": np.full(n, -800.0), "ninf": np.full(n, -np.inf)}[order]
    if order == "one":
        logw[n // 2] = 0.0
    got = ml.ml_resample_systematic(torch.from_numpy(logw).cuda(), seed=7, id_base=2).cpu().numpy()
    want = (np.full(n, -1) if order == "ninf"  # no positive weight
            else oracle.resample_systematic(logw, seed=7, id_base=2))
    assert np.array_equal(got, want)
