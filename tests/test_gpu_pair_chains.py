"""Edges of the pair kernel's tiling (three chains of 128-cell tiles per SM, tiles dealt out in
rounds over the SMs): grids of less than, exactly and just over one tile, one tile per chain
and one more with a ragged end. Every population of one step from random populations has to
meet the bound of tests/bf16_ref.py, derived from the BF16 rounding of the network's operands."""

import pytest

import lbm_inputs
from tests import gpu_util as G

pytestmark = pytest.mark.gpu


@pytest.fixture(scope="module", autouse=True)
def _cuda():
    torch = pytest.importorskip("torch")
    if not torch.cuda.is_available():
        pytest.skip("no CUDA device")
    G.P._abi.load()


# cells: 1, 127, 128, 129, 456 x 128 (every chain of 152 SMs one tile), 456 x 128 + 30
@pytest.mark.parametrize("shape", [(1, 1, 1), (1, 1, 127), (2, 8, 8), (3, 1, 43), (57, 32, 32), (2, 3, 9733)])
@pytest.mark.parametrize("storage", ["f16", "f32"])
def test_tile_edges(shape, storage):
    nu = 0.01
    ctx = G.make_ctx(shape, nu, "nco", storage=storage, net="bf16", theta=G.theta0())
    G.set_gpu_state(ctx, lbm_inputs.random_populations(shape, 31))
    G.check_bf16_step(ctx, nu, G.theta0(), storage=storage)
