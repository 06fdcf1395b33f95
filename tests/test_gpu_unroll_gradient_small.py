"""The gradient of a training step on grids of fewer 128-cell blocks than SMs, where the cotangent
of the moments is summed in parts (two here: 24^3 is 108 blocks): 150 unrolled steps of the
Taylor-Green octant against stored values, as tests/test_gpu_unroll_gradient.py at 32^3 and with
its tolerance.
"""

import os

import numpy as np
import pytest

import lbm_inputs
import paper_2412_08229_gb300 as P
from tests import gpu_util as G

pytestmark = pytest.mark.gpu
GOLDEN = os.path.join(os.path.dirname(os.path.abspath(__file__)), "golden", "unroll_gradient_octant24.txt")
N, STEPS, U0, RE, SEED = 24, 150, 0.045, 3000.0, 1


def gradient(seed):
    torch = pytest.importorskip("torch")
    rho, u = lbm_inputs.taylor_green_octant(N, U0)
    nu = lbm_inputs.reynolds_viscosity(U0, 2 * N, RE)
    theta = lbm_inputs.nco_parameters(seed).astype(np.float32)
    ctx = G.make_ctx((N, N, N), nu, "nco", bc="mirror", theta=theta)
    G.init_gpu(ctx, rho, u)
    P.lbm_record_begin(ctx, 20)
    P.lbm_step(ctx, STEPS)
    r = torch.empty((N, N, N), device="cuda")
    v = torch.empty((3, N, N, N), device="cuda")
    P.lbm_macroscopic(ctx, r, v)
    dtheta = torch.empty(theta.size, device="cuda")
    P.nco_backward(ctx, v - 0.9 * torch.from_numpy(u.astype(np.float32)).cuda(), None, dtheta, None)
    return dtheta.cpu().numpy()


def test_gradient_keeps_its_arithmetic_in_two_parts():
    ref = np.loadtxt(GOLDEN)
    got = gradient(SEED).astype(np.float64)
    assert np.linalg.norm(got - ref) <= 2e-6 * np.linalg.norm(ref)
