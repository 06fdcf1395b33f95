"""Steps replayed in chunks of sixteen (one graph launch each) against the same steps made one
call at a time: the same bits, from either buffer parity, at one step below, at and past the
chunk's size, with and without forcing.
"""

import numpy as np
import pytest

import lbm_inputs
import paper_2412_08229_gb300 as P
from tests import gpu_util as G

pytestmark = pytest.mark.gpu

SHAPE = (9, 10, 11)


def _run(op, net, forced, calls):
    theta = lbm_inputs.nco_parameters(0).astype(np.float32) if op == "nco" else None
    ctx = G.make_ctx(SHAPE, 0.01, op, net=net, theta=theta, forcing=dict(power=1e-6) if forced else None)
    G.set_gpu_state(ctx, lbm_inputs.random_populations(SHAPE, 7, 0.03, 0.04))
    rng = np.random.default_rng(3)
    phi, psi = rng.uniform(0, np.pi, (64, 16)), rng.uniform(0, 2 * np.pi, (64, 16))
    done = 0
    for n in calls:
        if forced:
            P.lbm_force_draws(ctx, phi[done:done + n], psi[done:done + n])
        P.lbm_step(ctx, n)
        done += n
    return G.gpu_state(ctx)


@pytest.mark.parametrize("op,net", [("bgk", "f32"), ("nco", "f32"), ("nco", "bf16")])
@pytest.mark.parametrize("forced", [False, True])
@pytest.mark.parametrize("calls", [(16,), (17,), (18, 33), (1, 34, 17)])
def test_chunks_are_the_single_steps(op, net, forced, calls):
    assert np.array_equal(_run(op, net, forced, calls), _run(op, net, forced, (1,) * sum(calls)))
