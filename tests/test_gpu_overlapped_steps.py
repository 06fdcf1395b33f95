"""Steps whose launches overlap (chunks of a graph, recorded steps) against the same steps made
one call at a time, at sizes where a step fills the GPU several times over and its last blocks run
beside the first ones of the next: the same bits, for every operator, storage and boundary that
is stepped so. 2^21 cells and one plane more are the two sides of the largest chunked grid.
"""

import numpy as np
import pytest

import lbm_inputs
import paper_2412_08229_gb300 as P
from tests import gpu_util as G

pytestmark = pytest.mark.gpu

RAGGED = (59, 61, 67)
BIG, BIGGER = (128, 128, 128), (129, 128, 128)


def _start(shape, op, storage, bc, deep):
    sizes = (27, 20, 20, 20, 4) if deep else (27, 20, 20, 4)
    theta = lbm_inputs.nco_parameters(0, sizes).astype(np.float32) if op == "nco" else None
    ctx = G.make_ctx(shape, 0.01, op, storage=storage, bc=bc, theta=theta)
    rng = np.random.default_rng(11)
    G.init_gpu(ctx, 1.0 + 0.01 * rng.standard_normal(shape).clip(-3, 3), 0.03 * rng.standard_normal((3,) + shape).clip(-3, 3))
    return ctx


CASES = [(RAGGED, op, st, "periodic", False) for op in ("bgk", "kbc", "reg") for st in ("f32", "f16")]
CASES += [(RAGGED, "bgk", "bf16", "mirror", False), (RAGGED, "kbc", "f32", "mirror", False),
          ((48, 48, 48), "bgk", "f32", "tgv_reduced", False), ((48, 48, 48), "reg", "f16", "tgv_reduced", False)]
CASES += [((37, 41, 39), "nco", "f32", "periodic", False), ((37, 41, 39), "nco", "f16", "mirror", True),
          ((31, 31, 31), "nco", "f32", "tgv_reduced", True)]
CASES += [(s, "bgk", "f32", "periodic", False) for s in (BIG, BIGGER)]


@pytest.mark.parametrize("shape,op,storage,bc,deep", CASES)
def test_one_call_is_the_single_steps(shape, op, storage, bc, deep):
    a, b = (_start(shape, op, storage, bc, deep) for _ in range(2))
    P.lbm_step(a, 40)
    for _ in range(40):
        P.lbm_step(b, 1)
    assert np.array_equal(G.gpu_state(a), G.gpu_state(b))


@pytest.mark.parametrize("shape,bc,deep", [((37, 41, 39), "periodic", False), ((19, 18, 17), "mirror", True),
                                           ((31, 31, 31), "tgv_reduced", False)])
def test_recorded_steps_are_the_single_steps(shape, bc, deep):
    a, b = (_start(shape, "nco", "f32", bc, deep) for _ in range(2))
    P.lbm_record_begin(a, 7)
    P.lbm_step(a, 20)
    for _ in range(20):
        P.lbm_step(b, 1)
    assert np.array_equal(G.gpu_state(a), G.gpu_state(b))
