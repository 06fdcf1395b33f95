"""The order of the FP32 network's group sum: the last hidden layer is summed over the 48
elements of O_h one after the other, as the oracle enumerates them. A long unrolled run amplifies
the last bit of a step until relu units switch, so another order of this sum is another
trajectory and another gradient.

The network is built so that the order decides the result. Its first hidden unit is on for a
single group element, the second layer turns it into L (2^25 <= L < 2^26, spacing 4) and adds 1
to it for every element, and the output layer takes L off again: 48 tau~ is the number of ones
that FP32 addition keeps, which is the position of that element (the ones before it, rounded to
the spacing; those after it fall below half of it). A position of 2 modulo 4 would be a tie, decided
by L's last bit. The rates show in the moments of order 3 and
more. Tolerance: one kept one is 1/48 in tau~ and at least 0.0045 in a rate (tau~ in [0, 1]); the
rates are read back from FP32 populations and moments of size 0.01, good to 1e-4; 1e-3 is allowed.
"""

import numpy as np
import pytest

import paper_2412_08229_gb300 as P
from oracle import lattice as L
from tests import gpu_util as G

pytestmark = pytest.mark.gpu

SHAPE = (3, 5, 7)  # 105 cells: four tiles, the last one partly empty


def _parameters(direction, deep):
    W1, b1 = np.zeros((20, 27)), np.zeros(20)
    W2, b2 = np.zeros((20, 20)), np.zeros(20)
    W3, b3 = np.zeros((4, 20)), np.zeros(4)
    W1[0, 1:4] = direction * 2.0 ** 10
    # between the largest and the second largest projection of the signed permutations of (1, 2, 4)
    b1[0] = -20.5 / 21.0 * (direction @ direction) * 2.0 ** 10
    W2[0, 0] = W2[1, 0] = 2.0 ** 25
    b2[0] = 1.0
    W3[:, 0], W3[:, 1] = 1.0, -1.0
    hidden = [W1, b1, W2, b2]
    if deep:
        hidden += [np.eye(20), np.zeros(20)]
    return np.concatenate([a.ravel() for a in hidden + [W3, b3]]).astype(np.float32)


@pytest.mark.parametrize("deep", [False, True], ids=["two", "deep"])
@pytest.mark.parametrize("element", [0, 3, 5, 12, 21, 31, 47])
def test_group_sum_runs_over_the_elements_in_order(element, deep):
    direction = 0.05 * np.array([1.0, 2.0, 4.0])
    perm, sign = L.moment_action_tables()
    m = np.zeros(27)
    m[0] = 1.0
    # the moments whose image under `element` points along `direction`
    for k in range(1, 4):
        m[perm[element, k]] = sign[element, k] * direction[k - 1]
    m[np.asarray(L.MOMENT_ORDER) >= 3] = 0.01
    theta = _parameters(direction, deep)
    images = sign * m[perm]
    on = np.maximum(images @ theta[:27].astype(np.float64) + float(theta[540]), 0.0)
    assert np.flatnonzero(on).tolist() == [element]
    # the sum as FP32 makes it, on the value of L that FP32 gives to within its spacing
    big = np.float32(on[element]) * np.float32(2.0 ** 25)
    assert 2.0 ** 25 <= big < 2.0 ** 26
    total = np.float32(0.0)
    for g in range(48):
        total = total + (big if g == element else np.float32(1.0))
    expected = 1.0 / (0.5 / (1.0 + np.exp(float(total - big) / 48.0)) + 0.5)

    ctx = G.make_ctx(SHAPE, 0.01, "nco", theta=theta)
    f = (L.M_INV @ m).astype(np.float32)
    G.set_gpu_state(ctx, np.broadcast_to(f[:, None, None, None], (27,) + SHAPE))
    start = G.to_oracle_f(G.gpu_state(ctx)) @ L.M.T
    P.lbm_step(ctx, 1)
    after = G.to_oracle_f(G.gpu_state(ctx)) @ L.M.T
    high = np.asarray(L.MOMENT_ORDER) >= 3
    rates = 1.0 - after[..., high] / start[..., high]
    assert np.abs(rates - expected).max() <= 1e-3
