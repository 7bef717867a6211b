"""F's extrapolated starts over hundreds of steps where the sweep's eigenvalues are negative (no
correlation, a Jacobi bound near the limit) or complex (drift above diffusion): the error of one
step must not grow in the next."""
import numpy as np
import pytest

import workloads as wl
from oracle import fd
from tests.gpu_util import FP32_FINE_TOL, oracle_fine, rel_err, start_state, to_gpu, to_np

pytestmark = pytest.mark.gpu


@pytest.fixture(scope="module")
def bs():
    import paper_2404_02521_gb300 as bs
    bs.load()
    yield bs
    bs.bs_set_option(bs.OPT_FINE_SWEEPS, 0)


def step_for(M, p, q):
    """The step size whose Gershgorin bound on this grid is q."""
    w = fd.stencil_weights(M, 4.0, p.sigma1, p.sigma2, p.rho, p.r)
    n = M - 1
    off = sum(np.abs(v[:n, :n]) for k, v in w.items() if k != (0, 0))
    diag = -w[(0, 0)][:n, :n]
    lo, hi = 0.0, 1e3
    for _ in range(100):
        mid = 0.5 * (lo + hi)
        lo, hi = (mid, hi) if np.max(mid * off / (1.0 + mid * diag)) <= q else (lo, mid)
    return lo


def propagated(bs, M, p, dtau, steps):
    import torch
    u0 = start_state(M, 4.0, p, "payoff")
    u = to_gpu(u0)
    g = bs.Grid(M, 4.0)
    bs.fine_propagate_batched(g, [p], [u], [u], [0.0], [dtau], steps)
    torch.cuda.synchronize()
    return rel_err(to_np(u), oracle_fine(M, 4.0, p, u0, 0.0, dtau, steps))


# three late sweeps lost every digit of the first three, two of the fourth; the others kept theirs.  In
# exact arithmetic the schedule leaves at most 2e-8 of the state's maximum in each.
@pytest.mark.parametrize("M,sigma1,sigma2,rho,r,q,steps", [
    (32, 0.3, 0.3, 0.0, 0.05, 0.72, 400), (64, 0.3, 0.3, 0.0, 0.05, 0.78, 400), (48, 0.3, 0.25, 0.2, 0.03, 0.75, 400),
    (32, 0.1, 0.1, 0.0, 1.0, 0.70, 400), (48, 0.1, 0.1, 0.3, 1.0, 0.60, 400), (33, 0.1, 0.15, 0.0, 3.0, 0.75, 200),
    (40, 0.3, 0.3, 0.0, 0.05, 0.705, 400), (40, 0.4, 0.4, 0.5, 1.0, 0.75, 400)])
def test_long_chains(bs, M, sigma1, sigma2, rho, r, q, steps):
    p = wl.Params(sigma1, sigma2, rho, r, payoff=wl.BASKET)
    assert propagated(bs, M, p, step_for(M, p, q), steps) <= FP32_FINE_TOL


# a forced count that extrapolated starts do not converge with starts every step from the previous
# increment, which leaves 3.6e-6 (three sweeps) and 1.2e-7 (two) in exact arithmetic
@pytest.mark.parametrize("count,M,sigma,r,q", [(3, 32, 0.3, 0.05, 0.75), (2, 32, 0.1, 1.0, 0.70)])
def test_forced_counts(bs, count, M, sigma, r, q):
    p = wl.Params(sigma, sigma, 0.0, r, payoff=wl.BASKET)
    bs.bs_set_option(bs.OPT_FINE_SWEEPS, count)
    try:
        assert propagated(bs, M, p, step_for(M, p, q), 400) <= 3.6e-6 + FP32_FINE_TOL
    finally:
        bs.bs_set_option(bs.OPT_FINE_SWEEPS, 0)
