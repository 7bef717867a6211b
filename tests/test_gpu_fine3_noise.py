"""Three-asset F on a state with every mode of the grid in it (white noise): the extrapolated starts
must not show beside the FP32 rounding."""
import types

import numpy as np
import pytest

import workloads as wl
from oracle import fd_nd

pytestmark = pytest.mark.gpu


# 40 steps at a Gershgorin bound of about 0.65: the rounding leaves 1e-6 of the state's norm; solves
# that stop at half of the extrapolated start's error left 6e-6
@pytest.mark.parametrize("M", [17, 24])
def test_white_noise_state(M):
    import torch
    import paper_2404_02521_gb300 as bs
    bs.load()
    p = types.SimpleNamespace(sigma=(0.3, 0.2, 0.25), rho=(0.5, -0.3, 0.2), r=0.05, strike=1.0,
                              w=(0.4, 0.35, 0.25), payoff=wl.BASKET)
    rho = np.array([[1.0, 0.5, -0.3], [0.5, 1.0, 0.2], [-0.3, 0.2, 1.0]])
    dtau = 6.0 / M ** 2

    def far(X, tau):
        return np.maximum(p.w[0] * X[0] + p.w[1] * X[1] + p.w[2] * X[2] - p.strike * np.exp(-p.r * tau), 0.0)

    noise = np.random.default_rng(M).standard_normal((M, M, M))
    u0 = (far(fd_nd.coords(M, 4.0, 3), 0.0) + noise).astype(np.float32)
    want = fd_nd.ImplicitEulerND(M, 4.0, p.sigma, rho, p.r, dtau, far).propagate(u0.astype(np.float64), 0.05, 40)
    u = torch.tensor(u0, device="cuda")
    bs.fine_propagate3(M, 4.0, p, [u], [u], [0.05], dtau, 40)
    torch.cuda.synchronize()
    got = u.cpu().double().numpy()
    assert np.linalg.norm(got - want) <= 3e-6 * np.linalg.norm(want)
