"""The captured steps of a context over several calls: chunks that come into use once enough
steps were asked for, and new weights between calls, which the captured steps read from device
memory; only another depth of the network captures anew. Against single steps, bit for bit.
"""

import time

import numpy as np
import pytest

import lbm_inputs
import paper_2412_08229_gb300 as P
from tests import gpu_util as G

pytestmark = pytest.mark.gpu
SHAPE = (9, 10, 11)


def _theta(seed, deep=False):
    return lbm_inputs.nco_parameters(seed, (27, 20, 20, 20, 4) if deep else (27, 20, 20, 4)).astype(np.float32)


def _run(op, net, forced, calls, single):
    ctx = G.make_ctx(SHAPE, 0.01, op, net=net, theta=_theta(0), forcing=dict(power=1e-6) if forced else None)
    G.set_gpu_state(ctx, lbm_inputs.random_populations(SHAPE, 7, 0.03, 0.04))
    phi, psi = lbm_inputs.forcing_draws(sum(calls))
    done = 0
    for n in calls:
        if forced:
            P.lbm_force_draws(ctx, phi[done:done + n], psi[done:done + n])
        for k in [1] * n if single else [n]:
            P.lbm_step(ctx, k)
        done += n
    return G.gpu_state(ctx)


@pytest.mark.parametrize("op,net", [("bgk", "f32"), ("nco", "f32"), ("nco", "bf16")])
@pytest.mark.parametrize("forced", [False, True])
@pytest.mark.parametrize("calls", [(70, 17, 33), (17, 17, 17, 17, 17, 17), (24, 25, 24, 49, 2, 81)])
def test_chunks_over_calls(op, net, forced, calls):
    assert np.array_equal(_run(op, net, forced, calls, False), _run(op, net, forced, calls, True))


@pytest.mark.parametrize("net", ["f32", "bf16", "bf16x3"])
@pytest.mark.parametrize("depths", [(False, False), (False, True), (True, False), (True, True)])
def test_new_weights_between_calls(net, depths):
    start = lbm_inputs.random_populations(SHAPE, 7, 0.03, 0.04)
    ctx = G.make_ctx(SHAPE, 0.01, "nco", net=net, theta=_theta(0, depths[0]))
    G.set_gpu_state(ctx, start)
    P.lbm_step(ctx, 52)
    P.nco_set_weights(ctx, _theta(1, depths[1]))
    G.set_gpu_state(ctx, start)
    P.lbm_step(ctx, 52)
    ref = G.make_ctx(SHAPE, 0.01, "nco", net=net, theta=_theta(1, depths[1]))
    G.set_gpu_state(ref, start)
    for _ in range(52):
        P.lbm_step(ref, 1)
    assert np.array_equal(G.gpu_state(ctx), G.gpu_state(ref))


def test_new_weights_capture_nothing():
    """Capturing a chunk and two single steps takes about 55 us; 25 us are allowed, on the shortest
    of 50 calls with and without new weights in turn."""
    torch = pytest.importorskip("torch")
    ctx = G.make_ctx((16, 16, 16), 0.01, "nco", theta=_theta(0))
    G.set_gpu_state(ctx, lbm_inputs.random_populations((16, 16, 16), 7, 0.03, 0.04))
    theta = torch.from_numpy(_theta(0)).cuda()
    best = [1.0, 1.0]
    for k in range(106):
        if k % 2:
            P.nco_set_weights(ctx, theta)
        torch.cuda.synchronize()
        t = time.perf_counter()
        P.lbm_step(ctx, 24)
        torch.cuda.synchronize()
        if k >= 6:
            best[k % 2] = min(best[k % 2], time.perf_counter() - t)
    assert best[1] - best[0] <= 25e-6
