"""A pointwise bias near the largest finite value: the parts that the 128 x 128 network adds it in stay
finite, as the bias does."""
import dataclasses

import numpy as np
import pytest

import workloads as wl
from tests.gpu_util import start_state, to_gpu, to_np
from tests.test_gpu_pino_cluster import rounded_network

pytestmark = pytest.mark.gpu


def test_bias_that_rounds_to_infinity_in_16_bits(tmp_path):
    import torch
    import paper_2404_02521_gb300 as bs
    from paper_2404_02521_gb300 import pino_io
    bs.load()
    arch = dataclasses.replace(wl.PinoArch(), layers=1, proj_hidden=16)
    w = wl.pino_random_weights(arch, seed=1, spectral_scale=8.0)
    # v = 1 in every channel; one channel's product is -3.3e38, the bias 3.4e38 (the largest BF16 value is 3.39e38)
    w = {k: np.zeros_like(v) for k, v in w.items()}
    w["lift_b"] += 1.0
    w["pw_w"][0, 0, :] = -3.3e38
    w["pw_b"] += np.float32(3.4e38)
    w["proj1_w"] += 1e-37
    w["proj2_w"] += 1.0 / 16
    path = str(tmp_path / "w.bin")
    pino_io.write_weights(path, w, arch.in_channels, arch.width, arch.modes_x, arch.modes_y, 1, 16)
    w, _ = pino_io.read_weights(path)
    M = 128
    net, g, p = bs.Pino(path), bs.Grid(M, 4.0), wl.basket_cfg1().params
    u = start_state(M, 4.0, p, "payoff")
    out = torch.empty((M, M), device="cuda")
    bs.coarse_propagate(g, bs.COARSE_PINO, net, p, to_gpu(u), out, 0.1, 1.0 / 64, 1)
    torch.cuda.synchronize()
    want, size = (v.cpu().numpy() for v in rounded_network(u, 4.0, 0.1, 1.0 / 64, p, w))
    d = (to_np(out) - u)[:-1, :-1] - want[:-1, :-1]
    assert np.max(np.abs(d)) <= 2.0 ** -8 * np.max(size)
