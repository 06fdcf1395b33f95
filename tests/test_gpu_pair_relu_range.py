"""The pair kernel's relu at the ends of the FP32 range: a unit of the second hidden layer at
minus infinity is off, and one above half of the largest float is itself. Each network is
compared with the same network scaled by powers of two to ordinary sizes: the same bits."""

import numpy as np
import pytest

import paper_2412_08229_gb300 as P
from oracle import lattice as L
from tests import gpu_util as G

pytestmark = pytest.mark.gpu
SHAPE = (3, 5, 7)


def _network(w2, w3):
    """One first-layer unit, 2.5 for the element that turns the flow's direction into (1, 2, 4)
    and 0 for the others, a constant one of 4, and a second-layer unit on each."""
    W1, b1 = np.zeros((20, 27)), np.zeros(20)
    W2, b2 = np.zeros((20, 20)), np.zeros(20)
    W3, b3 = np.zeros((4, 20)), np.array([0.1, 0.2, 0.3, 0.4])
    W1[0, 1:4] = 100.0 * np.array([1.0, 2.0, 4.0])  # 100 (21, next 20) times the state's 0.05
    b1[0], b1[1] = -102.5, 4.0
    W2[0, 0], W2[1, 1], W2[2, 1] = w2[0], w2[1], 0.25
    W3[:, 0], W3[:, 1], W3[:, 2] = w3, 0.5, 0.125
    return np.concatenate([a.ravel() for a in (W1, b1, W2, b2, W3, b3)]).astype(np.float32)


def _stepped(theta, storage):
    m = np.zeros(27)
    m[0], m[1:4], m[np.asarray(L.MOMENT_ORDER) >= 3] = 1.0, 0.05 * np.array([1.0, 2.0, 4.0]), 0.01
    f = (L.M_INV @ m).astype(np.float32)
    ctx = G.make_ctx(SHAPE, 0.01, "nco", storage=storage, net="bf16", theta=theta)
    G.set_gpu_state(ctx, np.broadcast_to(f[:, None, None, None], (27,) + SHAPE))
    P.lbm_step(ctx, 1)
    return G.gpu_state(ctx)


@pytest.mark.parametrize("storage", ["f32", "f16"])
def test_minus_infinity_is_off(storage):
    far = _stepped(_network((1.0, -3.0e38), 1.0), storage)  # 4 x -3e38: below the largest float
    near = _stepped(_network((1.0, -1.0), 1.0), storage)
    assert np.isfinite(far).all()
    assert np.array_equal(far, near)


@pytest.mark.parametrize("storage", ["f32", "f16"])
def test_half_the_largest_float_does_not_overflow(storage):
    far = _stepped(_network((2.0 ** 126, -1.0), 2.0 ** -126), storage)  # 2.5 x 2^126 > 2^127
    near = _stepped(_network((1.0, -1.0), 1.0), storage)
    assert np.isfinite(far).all()
    assert np.array_equal(far, near)
