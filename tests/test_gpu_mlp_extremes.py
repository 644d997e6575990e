"""SiLU of the tensor-core forward pass (rhi_mlp_forward) over its whole range, one value at a time: a
network whose first biases are z and whose other layers pass their input on computes
SiLU(SiLU(SiLU(z))) in BF16 steps, where exp(-z) overflows too, and an infinite activation stays
infinite.

Tolerance: three BF16 roundings (2^-9 each, of activations whose logarithmic derivative under SiLU is at most
|z| for z < 0 only in the first, FP32, one) stay below 2 %; below -89 the value is under 1e-37 in size."""
import numpy as np
import pytest

pytestmark = pytest.mark.gpu
IN, HID, OUT = 13, 64, 6


def _forward(W1, b1, W, W4, x):
    import paper_0901_1110_gb300 as rhi
    zero = np.zeros(HID)
    w = np.concatenate([W1.ravel(), b1, W.ravel(), zero, W.ravel(), zero, W4.ravel(), np.zeros(OUT),
                        np.zeros(IN), np.ones(IN)]).astype(np.float32)
    s = rhi.Solver(2, 2, 2, 1e22, rhi.rhi_params_default(1))
    s.mlp_set_weights(w)
    Y = s.mlp_forward(np.full((33, IN), x, dtype=np.float32))
    s.close()
    return Y


def _silu(z):
    return z / (1.0 + np.exp(-z)) if z > -700.0 else 0.0


@pytest.mark.parametrize("z", [-3e38, -1e38, -1e30, -1e4, -100.0, -89.5, -88.5, -88.0, -60.0, -20.0, -1.0, 0.0, 0.5, 5.0,
                               80.0, 100.0, 1e30, 3e38])
def test_chain_of_silu(z):
    Y = _forward(np.zeros((HID, IN)), np.full(HID, z), np.eye(HID), np.eye(OUT, HID), 0.0)
    want = _silu(_silu(_silu(float(np.float32(z)))))
    assert np.all(np.abs(Y - want) <= 0.02 * abs(want) + 1e-37), (Y[0], want)


def test_infinite_activation_stays_infinite():
    Y = _forward(np.ones((HID, IN)), np.zeros(HID), np.ones((HID, HID)), np.ones((OUT, HID)), np.inf)
    assert np.all(np.isposinf(Y)), Y[0]
