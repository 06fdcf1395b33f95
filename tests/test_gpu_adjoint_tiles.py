"""The adjoint kernel's tiles (32 cells with the two-layer network, 16 with the third hidden
layer) at the edges of their range: fewer cells than a tile, exactly one, one more, and ragged
boxes whose last tile is partly empty; against autograd of the FP64 PyTorch restatement of the
oracle. Tolerance: 1e-3 relative, the adjoint tests' bound for FP32 against FP64 (the relu
units that switch between the two precisions dominate it).
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

NU, STEPS = 0.01, 3


@pytest.mark.parametrize("sizes", [(27, 20, 20, 4), (27, 20, 20, 20, 4)], ids=["two", "deep"])
@pytest.mark.parametrize("shape", [(1, 1, 1), (2, 2, 2), (4, 4, 2), (4, 2, 2), (3, 11, 1), (17, 1, 1), (5, 7, 9)])
def test_adjoint_at_tile_edges(shape, sizes):  # shape: (nz, ny, nx)
    f0 = lbm_inputs.random_populations(shape, 23).astype(np.float32)
    theta = lbm_inputs.nco_parameters(0, sizes).astype(np.float32)
    rng = np.random.default_rng(5)
    a = rng.standard_normal((3,) + shape).astype(np.float32)
    b = rng.standard_normal(shape).astype(np.float32)

    th = torch.tensor(theta.astype(np.float64), requires_grad=True)
    ft = torch.tensor(np.moveaxis(f0, 0, -1).astype(np.float64), requires_grad=True)
    f = T.run(ft, col.tau_from_nu(NU), th, STEPS, bc="periodic", sizes=sizes)
    a64, b64 = torch.tensor(np.moveaxis(a, 0, -1).astype(np.float64)), torch.tensor(b.astype(np.float64))
    ((T.velocity(f) * a64).sum() + (f.sum(-1) * b64).sum()).backward()

    ctx = G.make_ctx(shape, NU, "nco", theta=theta)
    G.set_gpu_state(ctx, f0)
    P.lbm_record_begin(ctx, 2)
    P.lbm_step(ctx, STEPS)
    dtheta = torch.zeros(theta.size, device="cuda")
    df0 = torch.zeros((27,) + shape, device="cuda")
    P.nco_backward(ctx, torch.from_numpy(a).cuda(), torch.from_numpy(b).cuda(), dtheta, df0)

    def rel(x, y):
        return float(np.linalg.norm(x - y) / np.linalg.norm(y))

    assert rel(np.moveaxis(df0.cpu().numpy().astype(np.float64), 0, -1), ft.grad.numpy()) <= 1e-3
    got, ref = dtheta.cpu().numpy().astype(np.float64), th.grad.numpy()
    if np.prod(shape) == 1:  # mass and momentum of one cell do not depend on the network: no relative error
        assert np.linalg.norm(got) <= 2.0 ** -23 * np.linalg.norm(np.append(a.ravel(), b.ravel()))
    else:
        assert rel(got, ref) <= 1e-3
