"""Three-asset F's extrapolated starts over many steps where the sweep's eigenvalues are negative (no
correlation) or complex (drift above diffusion)."""
import types

import numpy as np
import pytest

import workloads as wl
from oracle import fd_nd
from tests.gpu_util import FP32_FINE_TOL, rel_err

pytestmark = pytest.mark.gpu


def step_for(M, sigma, C, r, q):
    """The step size whose Gershgorin bound on this grid is q."""
    inner = (slice(0, M - 1),) * 3
    w = fd_nd.stencil_weights(M, 4.0, sigma, C, r)
    off = sum(np.abs(v[inner]) for k, v in w.items() if k != (0, 0, 0))
    diag = -w[(0, 0, 0)][inner]
    lo, hi = 0.0, 1e3
    for _ in range(100):
        mid = 0.5 * (lo + hi)
        lo, hi = (mid, hi) if np.max(mid * off / (1.0 + mid * diag)) <= q else (lo, mid)
    return lo


def setup(M, sigma, rho, r):
    p = types.SimpleNamespace(sigma=sigma, rho=rho, r=r, strike=1.0, w=(0.4, 0.35, 0.25), payoff=wl.BASKET)
    C = np.array([[1.0, rho[0], rho[1]], [rho[0], 1.0, rho[2]], [rho[1], rho[2], 1.0]])

    def far(X, tau):
        return np.maximum(p.w[0] * X[0] + p.w[1] * X[1] + p.w[2] * X[2] - p.strike * np.exp(-r * tau), 0.0)

    return p, C, far, far(fd_nd.coords(M, 4.0, 3), 0.0).astype(np.float32)


@pytest.mark.parametrize("M,sigma,rho,r,q", [
    (16, (0.1, 0.1, 0.1), (0.0, 0.0, 0.0), 1.0, 0.70), (14, (0.1, 0.15, 0.1), (0.2, 0.0, 0.1), 3.0, 0.60),
    (16, (0.3, 0.3, 0.3), (0.0, 0.0, 0.0), 0.05, 0.72), (15, (0.3, 0.2, 0.25), (0.5, -0.3, 0.2), 0.05, 0.78)])
def test_long_chains(M, sigma, rho, r, q):
    import torch
    import paper_2404_02521_gb300 as bs
    bs.load()
    p, C, far, u0 = setup(M, sigma, rho, r)
    dtau, steps = step_for(M, sigma, C, r, q), 200
    want = fd_nd.ImplicitEulerND(M, 4.0, sigma, C, r, dtau, far).propagate(u0.astype(np.float64), 0.0, steps)
    u = torch.tensor(u0, device="cuda")
    bs.fine_propagate3(M, 4.0, p, [u], [u], [0.0], dtau, steps)
    torch.cuda.synchronize()
    assert rel_err(u.cpu().double().numpy(), want) <= FP32_FINE_TOL


# drift above diffusion on grids whose eigenvalues come near the bound: two late sweeps grow the error by
# 1.05 (32^3) to 1.15 (64^3) per step.  The same steps in calls of 25, which end before the late schedule,
# are the reference.
@pytest.mark.parametrize("M,sigma,r,steps", [(64, 0.05, 1.0, 300), (48, 0.1, 3.0, 400)])
def test_complex_eigenvalues(M, sigma, r, steps):
    import torch
    import paper_2404_02521_gb300 as bs
    bs.load()
    p, C, _, u0 = setup(M, (sigma,) * 3, (0.0, 0.0, 0.0), r)
    dtau = step_for(M, (sigma,) * 3, C, r, 0.70)
    whole, parts = torch.tensor(u0, device="cuda"), torch.tensor(u0, device="cuda")
    bs.fine_propagate3(M, 4.0, p, [whole], [whole], [0.0], dtau, steps)
    for s in range(0, steps, 25):
        bs.fine_propagate3(M, 4.0, p, [parts], [parts], [s * dtau], dtau, 25)
    torch.cuda.synchronize()
    assert rel_err(whole.cpu().double().numpy(), parts.cpu().double().numpy()) <= FP32_FINE_TOL
