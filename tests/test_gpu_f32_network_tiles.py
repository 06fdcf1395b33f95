"""The FP32 network step's tiles of 32 cells at the edges of their range (fewer cells than a
tile, exactly one, one more, ragged boxes, more tiles than SMs), both depths and every storage,
against the FP64 oracle. Tolerance: 1e-5 relative for FP32 storage and for 16-bit storage the
rounding of f - w (its largest value, at most 1, times 2^-11 or 2^-8 relative, halved by
rounding to nearest) on top of it.
"""

import numpy as np
import pytest

import lbm_inputs
import paper_2412_08229_gb300 as P
from oracle import collision as col
from oracle import stepper as S
from tests import gpu_util as G

pytestmark = pytest.mark.gpu

NU = 0.02
DEEP = (27, 20, 20, 20, 4)


@pytest.mark.parametrize("storage", ["f32", "f16", "bf16"])
@pytest.mark.parametrize("sizes", [(27, 20, 20, 4), DEEP], ids=["two", "deep"])
@pytest.mark.parametrize("shape", [(1, 1, 1), (4, 4, 2), (3, 11, 1), (5, 7, 9), (19, 18, 17)])
def test_step_at_tile_edges(shape, sizes, storage):
    theta = lbm_inputs.nco_parameters(0, sizes).astype(np.float32)
    ctx = G.make_ctx(shape, NU, "nco", storage=storage, theta=theta)
    G.set_gpu_state(ctx, lbm_inputs.random_populations(shape, 41))
    start = G.to_oracle_f(G.gpu_state(ctx))
    P.lbm_step(ctx, 1)
    got = G.to_oracle_f(G.gpu_state(ctx))
    ref = S.Simulation(start, col.tau_from_nu(NU), op="nco", theta=theta.astype(np.float64), sizes=sizes).step(1).f
    dev = np.abs(ref - col.equilibrium(np.ones(1), np.zeros((1, 3)))[0]).max()
    tol = 1e-5 * np.abs(ref).max() + {"f32": 0.0, "f16": 2.0 ** -11, "bf16": 2.0 ** -8}[storage] * dev
    assert np.abs(got - ref).max() <= tol
