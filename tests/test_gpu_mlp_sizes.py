"""Prediction and gradients of the warm-start network at the edges of their
sample groups and staging, against the FP64 oracle."""
from concurrent.futures import ThreadPoolExecutor

import numpy as np
import pytest

from oracle import mlp as ref
from paper_1204_4098_gb300 import lbm

pytestmark = pytest.mark.gpu


def network(seed):
    theta = ref.init_params(seed) + 0.05 * np.random.default_rng(seed).standard_normal(
        ref.N_PARAMS)
    return theta.astype(np.float32)


# groups of 16 samples; mapped staging up to 4096, device staging up to 2^18
@pytest.mark.parametrize("sizes", [(1, 15, 16, 17, 4096, 33), (4097, 3, 20000, 5000, 262144),
                                   (262145, 16)])
def test_predict_sizes(sizes):
    theta = network(3)
    net = lbm.MLP(theta)
    for n in sizes:
        X = np.random.default_rng(n).uniform(-1, 1, (n, 4)).astype(np.float32)
        want, _ = ref.forward(theta.astype(np.float64), X)
        # 64-term FP32 sums of O(1) terms through two layers
        assert np.max(np.abs(net.predict(X) - want)) < 1e-5


# minibatches that leave CTAs of the training cluster without samples (16 each)
@pytest.mark.parametrize("n", [1, 15, 16, 17, 31, 33, 100, 127, 128])
def test_gradient_sizes(n):
    theta = network(4)
    rng = np.random.default_rng(n)
    X, T = rng.uniform(-1, 1, (n, 4)), rng.standard_normal((n, 3))
    loss, g = lbm.MLP(theta).gradient(X, T)
    want_loss, want = ref.gradient(theta.astype(np.float64), X.astype(np.float32),
                                   T.astype(np.float32))
    assert loss == pytest.approx(want_loss, rel=1e-5)
    assert np.max(np.abs(g - want)) <= 2e-5 * np.max(np.abs(want)) + 1e-8


# several threads predicting with one network: none gets another's staging
def test_predict_from_several_threads():
    net = lbm.MLP(network(5))
    jobs = [np.random.default_rng(k).uniform(-1, 1, (n, 4)).astype(np.float32)
            for k, n in enumerate([17, 300, 4096, 5000, 1, 20000, 64, 4097] * 8)]
    want = [net.predict(X) for X in jobs]
    with ThreadPoolExecutor(8) as pool:
        for got, w in zip(pool.map(net.predict, jobs), want):
            assert np.array_equal(got, w)
