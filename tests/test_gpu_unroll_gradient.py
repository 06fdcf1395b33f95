"""The gradient of a training step at its real horizon: 32^3 Taylor-Green octant, 200 unrolled
steps, against stored values. An unrolled gradient is a sum with cancellations behind a long
linear sweep, so roundings of the step or of the cotangents that come out differently move it by
1e-5 and more: the step's and the sweep's arithmetic have to stay what they are, bit for bit.
The stored values were computed by one thread per cell, which fixes that arithmetic: the group
sum element by element, the cotangent of a moment as the relaxation's part plus the network's,
permutation by permutation and unit by unit.

Tolerance 2e-6 of the 2-norm: only the parameter sums over cells, columns and permutations may
be grouped in another way, in FP32 within a tile (2^-24 per sum, about four sums deep, against
terms that cancel to a tenth of their size) and in FP64 beyond it. Against FP64 the gradient is
off by 0.2e-5 to 4.7e-5 from run to run (relu units that switch); 1e-4 is allowed.
"""

import os

import numpy as np
import pytest

import lbm_inputs
import paper_2412_08229_gb300 as P
from tests import gpu_util as G

pytestmark = pytest.mark.gpu
GOLDEN = os.path.join(os.path.dirname(os.path.abspath(__file__)), "golden", "unroll_gradient_octant32.txt")
N, STEPS, U0, RE, SEEDS = 32, 200, 0.045, 3000.0, (0, 3)


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
    du = v - 0.9 * torch.from_numpy(u.astype(np.float32)).cuda()
    P.nco_backward(ctx, du, None, dtheta, None)
    return dtheta.cpu().numpy()


@pytest.mark.parametrize("seed", SEEDS)
def test_gradient_keeps_its_arithmetic(seed):
    rows = np.loadtxt(GOLDEN)
    ref, exact = rows[SEEDS.index(seed)], rows[len(SEEDS) + SEEDS.index(seed)]
    got = gradient(seed).astype(np.float64)
    assert np.linalg.norm(got - ref) <= 2e-6 * np.linalg.norm(ref)
    assert np.linalg.norm(got - exact) <= 1e-4 * np.linalg.norm(exact)
