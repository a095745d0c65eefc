"""Training in one cluster of CTAs at the edges of its rows: mini-batches around
128 rows a CTA and up to eight CTAs (the last one beyond, which trains step by
step).  The sum of squared residuals and the Adam step of the first training
step against the library's own gradient of the same rows (regc_surrogate_
gradient_bf16, one CTA per 128 rows), and a run in two calls equals one call."""
import numpy as np
import pytest

import workloads as W
from oracle import surrogate as SG
from paper_1908_11118_gb300 import Regc
from paper_1908_11118_gb300 import build as B
from paper_1908_11118_gb300.regc import surrogate_gradient

pytestmark = pytest.mark.gpu


@pytest.fixture(scope="module", autouse=True)
def built():
    B.build()


@pytest.mark.parametrize("batch", [1, 31, 127, 128, 129, 300, 1023, 1024, 1025])
def test_cluster_training_shapes(batch):
    p = W.fcc100_small(L=2, M=2, seed=9)
    rng = np.random.default_rng(batch)
    X = rng.gamma(1.0, 0.5, (700, 16)).astype(np.float32)
    y = (X @ rng.normal(size=16) - 1.0).astype(np.float32)
    th = SG.init_params(3, scale=1.0).astype(np.float32)
    key = (int(p.seed) & 0xFFFFFFFF, int(p.seed) >> 32)
    rows = SG.batch_rows(1, batch, len(y), key)
    loss, grad = surrogate_gradient(th, X[rows], y[rows], tensor_cores=True)
    lr = 1e-3

    def trained(*calls):
        g = Regc(p)
        g.surrogate_set(th)
        g.surrogate_set_dataset(X, y, capacity=1024)
        return np.concatenate([g.surrogate_train(k, batch, lr) for k in calls]), g.surrogate_get()

    l1, t1 = trained(1)
    # the same sums in the same order: the loss up to its division by the batch
    assert abs(l1[0] - loss) <= 1e-6 * abs(loss)
    # the first Adam step is lr g / (|g| + eps): a few roundings of the update
    # and one of theta away
    step = -lr * grad.astype(np.float64) / (np.abs(grad.astype(np.float64)) + 1e-8)
    assert np.all(np.abs(t1 - (th + step)) <= 2e-5 * lr + 2.0 ** -23 * np.abs(th))
    la, ta = trained(7)
    lb, tb = trained(3, 4)
    assert np.array_equal(la, lb) and np.array_equal(ta, tb)
    assert np.isfinite(ta).all() and not np.array_equal(ta, t1)


@pytest.mark.parametrize("layer", [0, 1, 2])
def test_cluster_training_far_units(layer):
    """Units far below zero (x < -80, and where exp(-x) overflows), whose SiLU
    derivatives take the general form: in layer 1, layer 2 or both, next to
    ordinary units.  The same comparison as above."""
    p = W.fcc100_small(L=2, M=2, seed=9)
    rng = np.random.default_rng(layer)
    X = rng.gamma(1.0, 0.5, (300, 16)).astype(np.float32)
    y = (X @ rng.normal(size=16) - 1.0).astype(np.float32)
    th = SG.init_params(3, scale=1.0).astype(np.float32)
    for on, b in ((layer != 1, 1024), (layer != 0, 1024 + 64 + 4096)):   # b1, b2
        if on:
            th[b:b + 64:4] = -84.0
            th[b + 1:b + 64:4] = -200.0
    key = (int(p.seed) & 0xFFFFFFFF, int(p.seed) >> 32)
    rows = SG.batch_rows(1, 200, len(y), key)
    loss, grad = surrogate_gradient(th, X[rows], y[rows], tensor_cores=True)
    g = Regc(p)
    g.surrogate_set(th)
    g.surrogate_set_dataset(X, y, capacity=512)
    l1, t1 = g.surrogate_train(1, 200, 1e-3), g.surrogate_get()
    assert abs(l1[0] - loss) <= 1e-6 * abs(loss)
    step = -1e-3 * grad.astype(np.float64) / (np.abs(grad.astype(np.float64)) + 1e-8)
    assert np.all(np.abs(t1 - (th + step)) <= 2e-5 * 1e-3 + 2.0 ** -23 * np.abs(th))
    assert np.isfinite(t1).all()
