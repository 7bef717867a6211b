"""The training loss's PDE term on the wide tiles that a batch of many tiles runs on: a tile's width and one
node on either side of it, and two states of many tiles, against the oracle."""
import numpy as np
import pytest

import workloads as wl
from oracle import fd, physics
from tests.gpu_util import to_gpu, to_np

pytestmark = pytest.mark.gpu

REL_TOL = 1e-4   # an FP32 residual that cancels by up to two decimal digits: 16 * 6e-8 * 100


# 32-node tiles from 304 of them in a launch: 32, 20, 16 and 2 samples of 16, 16, 25 and 324 tiles; 40 samples
# of 16 tiles are a launch of 32 on wide tiles and one of 8 on narrow ones
@pytest.mark.parametrize("M,B", [(128, 32), (127, 20), (129, 16), (545, 2), (128, 40)])
def test_wide_tiles(M, B):
    import torch
    import paper_2404_02521_gb300 as bs
    bs.load()
    rng = np.random.default_rng([M, B])
    params = [wl.random_params(rng, k % 2) for k in range(B)]
    dtaus = [float(rng.uniform(0.002, 0.08)) for _ in range(B)]
    prev = [wl.random_field(rng, M).astype(np.float32) for _ in range(B)]
    pred = [(v + dt * wl.random_field(rng, M)).astype(np.float32) for v, dt in zip(prev, dtaus)]
    loss = torch.empty(B, dtype=torch.float64, device="cuda")
    grads = [torch.full((M, M), float("nan"), device="cuda") for _ in range(B)]
    bs.pino_physics_loss(bs.Grid(M, 4.0), params, [to_gpu(a) for a in pred], [to_gpu(a) for a in prev], dtaus,
                         loss, grads)
    torch.cuda.synchronize()
    for b in range(B):
        w = fd.stencil_weights(M, 4.0, params[b].sigma1, params[b].sigma2, params[b].rho, params[b].r)
        u1, u0 = pred[b].astype(np.float64), prev[b].astype(np.float64)
        want, gw = physics.loss(u1, u0, dtaus[b], w), physics.loss_grad(u1, u0, dtaus[b], w)
        assert abs(float(loss[b]) - want) <= REL_TOL * want, b
        assert np.max(np.abs(to_np(grads[b]) - gw)) <= REL_TOL * np.max(np.abs(gw)), b
