"""The surrogate network's kernels at the edges of their tiles: batches of one
sample, just below, at and above 16, 32, 128, 256 and 257 samples, against a
64-bit evaluation with the same rounding points of the weights and layer
inputs (oracle.mlp, quant=True); and a training call, recorded and replayed,
against the same steps taken one by one.

Predictions: FP32 accumulation over 512 products per layer and four layers,
4 * 512 * 2^-24 = 1.2e-4 at the very worst, random signs leave about its
square root; 1e-5 is asked.  Gradients carry one-term bf16 error signals
(2^-9 per value): 2 % of a layer's norm, as the repository's gradient test."""
import numpy as np
import pytest

import oracle.mlp as om
from paper_1610_06749_gb300 import binding as B
from paper_1610_06749_gb300 import synth

pytestmark = pytest.mark.gpu


@pytest.fixture(scope="module", autouse=True)
def _lib():
    from paper_1610_06749_gb300 import build
    build.build()
    B.lib()


def _net(members, max_batch):
    theta = synth.mlp_init(21, members).astype(np.float32)
    h = B.it_mlp_create(members, max_batch)
    for m in range(members):
        B.it_mlp_set_params(h, m, theta[m])
    return h, theta


def _data(n):
    X = 4.0 * synth.uniform01(31, 6 * n).reshape(n, 6) - 2.0
    return X, synth.uniform01(32, n)


@pytest.mark.parametrize("n", [1, 15, 16, 17, 31, 33, 127, 129, 255, 256, 257])
def test_batches_at_tile_edges(n):
    h, theta = _net(2, 300)
    try:
        X, y = _data(n)
        X = X.astype(np.float32).astype(np.float64)
        _, _, per = B.it_mlp_predict(h, 2, X)
        loss, g = B.it_mlp_loss_grad(h, 2, X, y)
        for m in range(2):
            f, _ = om.forward(theta[m].astype(np.float64), X, quant=True)
            assert np.max(np.abs(per[:, m] - f)) <= 1e-5
            lo, go = om.loss_and_grad(theta[m].astype(np.float64), X, y, quant=True)
            assert abs(loss[m] - lo) <= 1e-5
            assert np.linalg.norm(g[m] - go) <= 0.02 * np.linalg.norm(go)
    finally:
        B.it_mlp_destroy(h)


@pytest.mark.parametrize("samples,batch", [(160, 16), (165, 33), (300, 256)])
def test_training_equals_its_steps_one_by_one(samples, batch):
    # a call of eight or more steps is recorded and replayed: bitwise the
    # gradient and Adam calls on the same mini-batches
    X, y = _data(samples)
    X, y = X.astype(np.float32).astype(np.float64), y.astype(np.float32).astype(np.float64)
    epochs = 2
    mask, st = (1 << 64) - 1, (7 + 0x9E3779B97F4A7C15) & ((1 << 64) - 1)
    res = []
    h, _ = _net(1, batch)
    try:
        B.it_mlp_set_data(h, X, y)
        B.it_mlp_train(h, epochs, batch, 1e-3, 7)
        res.append(B.it_mlp_get_params(h, 0))
    finally:
        B.it_mlp_destroy(h)
    h, _ = _net(1, batch)
    try:
        for _ in range(epochs):
            p = list(range(samples))
            for i in range(samples - 1, 0, -1):       # SplitMix64 Fisher-Yates
                st = (st + 0x9E3779B97F4A7C15) & mask
                v = ((st ^ (st >> 30)) * 0xBF58476D1CE4E5B9) & mask
                v = ((v ^ (v >> 27)) * 0x94D049BB133111EB) & mask
                j = (v ^ (v >> 31)) % (i + 1)
                p[i], p[j] = p[j], p[i]
            for b in range(samples // batch):
                idx = p[b * batch:(b + 1) * batch]
                B.it_mlp_loss_grad(h, 1, X[idx], y[idx])
                B.it_mlp_adam_step(h, 1e-3)
        res.append(B.it_mlp_get_params(h, 0))
    finally:
        B.it_mlp_destroy(h)
    assert np.array_equal(res[0], res[1])
