"""The adjoint's blocks over more than one tile (a block per SM walks the tiles of 32 cells, or 16
with the third hidden layer, and keeps its gradient sums from one to the next), with a ragged end,
on every boundary, and partly empty tiles on the mirror and the reduced Taylor-Green domain;
against autograd of the FP64 PyTorch restatement of the oracle. Tolerance: 1e-3 relative, the
adjoint tests' bound for FP32 against FP64 (the relu units that switch between the two precisions
dominate it).
"""

import numpy as np
import pytest

import lbm_inputs
import paper_2412_08229_gb300 as P
from oracle import collision as col
from tests import gpu_util as G

pytestmark = pytest.mark.gpu
torch = pytest.importorskip("torch")
from oracle import torch_ref as T  # noqa: E402

NU, STEPS = 0.01, 2
TWO, DEEP = (27, 20, 20, 4), (27, 20, 20, 20, 4)

# cells: 5814 (182 tiles of 32), 2660 (167 of 16), 5832 and 2744 (reduced), more than 152 tiles each; then 27, 125, 343
CASES = [((17, 18, 19), "periodic", TWO), ((17, 18, 19), "mirror", TWO), ((18, 18, 18), "tgv_reduced", TWO),
         ((14, 10, 19), "periodic", DEEP), ((14, 10, 19), "mirror", DEEP), ((14, 14, 14), "tgv_reduced", DEEP)]
CASES += [((n, n, n), bc, s) for n in (3, 5, 7) for bc in ("mirror", "tgv_reduced") for s in (TWO, DEEP)]


@pytest.mark.parametrize("shape,bc,sizes", CASES)
def test_adjoint_over_many_tiles(shape, bc, sizes):
    f0 = lbm_inputs.random_populations(shape, 29).astype(np.float32)
    theta = lbm_inputs.nco_parameters(0, sizes).astype(np.float32)
    rng = np.random.default_rng(8)
    a = rng.standard_normal((3,) + shape).astype(np.float32)
    b = rng.standard_normal(shape).astype(np.float32)

    th = torch.tensor(theta.astype(np.float64), requires_grad=True)
    ft = torch.tensor(np.moveaxis(f0, 0, -1).astype(np.float64), requires_grad=True)
    f = T.run(ft, col.tau_from_nu(NU), th, STEPS, bc=bc, sizes=sizes)
    a64, b64 = torch.tensor(np.moveaxis(a, 0, -1).astype(np.float64)), torch.tensor(b.astype(np.float64))
    ((T.velocity(f) * a64).sum() + (f.sum(-1) * b64).sum()).backward()

    ctx = G.make_ctx(shape, NU, "nco", bc=bc, theta=theta)
    G.set_gpu_state(ctx, f0)
    P.lbm_record_begin(ctx, 2)
    P.lbm_step(ctx, STEPS)
    dtheta = torch.zeros(theta.size, device="cuda")
    df0 = torch.zeros((27,) + shape, device="cuda")
    P.nco_backward(ctx, torch.from_numpy(a).cuda(), torch.from_numpy(b).cuda(), dtheta, df0)

    def rel(x, y):
        return float(np.linalg.norm(x - y) / np.linalg.norm(y))

    assert rel(np.moveaxis(df0.cpu().numpy().astype(np.float64), 0, -1), ft.grad.numpy()) <= 1e-3
    assert rel(dtheta.cpu().numpy().astype(np.float64), th.grad.numpy()) <= 1e-3
