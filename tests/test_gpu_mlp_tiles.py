"""The training kernel's tiles (32 samples per block, at most 304 blocks) against the FP64 oracle at the
sizes where they can go wrong: one sample, a tile less or more one, one tile per block and one sample
more, and a minibatch size that leaves a ragged last batch.

Tolerance: dot products of at most 64 FP32 terms lose at most 64 x 2^-24 = 3.8e-6 of the sum of their
terms' sizes; three layers forward and three back add up to 2.3e-5."""
import numpy as np
import pytest

from oracle import mlp as om
from paper_0901_1110_gb300 import inputs

pytestmark = pytest.mark.gpu
TOL = 2.5e-5


def _data(rows, seed):
    rng = np.random.default_rng(seed)
    X = rng.standard_normal((rows, om.NIN))
    w = om.unpack(om.init_weights(seed))
    w["mean"], w["scale"] = rng.uniform(-2, 2, om.NIN), rng.uniform(0.5, 3.0, om.NIN)
    X = X * w["scale"] + w["mean"]
    return X.astype(np.float32), rng.standard_normal((rows, om.NOUT)).astype(np.float32), om.pack(w).astype(np.float32)


def _solver(rhi):
    return rhi.Solver(2, 2, 2, inputs.KPC, rhi.rhi_params_default(1))


@pytest.mark.parametrize("rows", [1, 31, 32, 33, 304 * 32, 304 * 32 + 1])
def test_gradient_at_tile_edges(rows):
    import paper_0901_1110_gb300 as rhi
    X, Y, w = _data(rows, 3)
    s = _solver(rhi)
    s.mlp_set_weights(w)
    loss, g = s.mlp_loss_grad(X, Y)
    lr, gr = om.loss_and_grad(w.astype(np.float64), X.astype(np.float64), Y.astype(np.float64))
    assert abs(loss / lr - 1) <= TOL
    assert np.linalg.norm(g - gr) <= TOL * np.linalg.norm(gr)
    assert not g[-2 * om.NIN:].any()


def test_ragged_last_minibatch_follows_adam():
    """Three steps of 100, 100 and 37 samples: Adam restated in FP64.  Its first step is the sign of each
    gradient entry, so weights are compared in the mean (2-norm), where entries next to 0 count little."""
    import torch

    import paper_0901_1110_gb300 as rhi
    X, Y, w = _data(237, 5)
    s = _solver(rhi)
    s.mlp_set_weights(w)
    s.mlp_train(torch.from_numpy(X).cuda(), torch.from_numpy(Y).cuda(), epochs=1, batch=100, lr=1e-3)
    v, m1, m2 = w.astype(np.float64), 0.0, 0.0
    for t, a in enumerate((0, 100, 200), 1):
        _, g = om.loss_and_grad(v, X[a:a + 100].astype(np.float64), Y[a:a + 100].astype(np.float64))
        m1, m2 = 0.9 * m1 + 0.1 * g, 0.999 * m2 + 0.001 * g * g
        up = 1e-3 * (m1 / (1 - 0.9 ** t)) / (np.sqrt(m2 / (1 - 0.999 ** t)) + 1e-8)
        up[-2 * om.NIN:] = 0.0
        v = v - up
    assert np.linalg.norm(s.mlp_get_weights() - v) <= TOL * np.linalg.norm(v - w)
