"""Cash-or-nothing far-field data on both sides of the argument from which the bivariate normal's
correlation integral is left out."""
import numpy as np
import pytest

import workloads as wl
from oracle import closed_forms as cf

pytestmark = pytest.mark.gpu

# Phi's slope times the rounding of its argument (0.24 x 3e-7), 2 ulp of Phi, and twenty exponentials
# of 2 ulp with weights that sum to 1 / 6: below 1e-6 of the cash
TOL = 1e-6


@pytest.mark.parametrize("rho", [-0.9, -0.3, 0.5, 0.9])
@pytest.mark.parametrize("sigma1,sigma2,r,tau", [(0.3, 0.3, 1.0, 1.0), (0.3, 0.3, 1.0, 0.2), (0.16, 0.5, 0.0, 1.0),
                                                 (0.5, 0.8, 0.05, 1.0), (0.165, 0.163, 0.0, 1.0)])
def test_edges(rho, sigma1, sigma2, r, tau):
    import torch
    import paper_2404_02521_gb300 as bs
    bs.load()
    M, xmax = 61, 300.0
    p = wl.Params(sigma1, sigma2, rho, r, 1.0, 100.0, payoff=wl.CASH_OR_NOTHING, strike2=100.0, cash=1.0)
    u = torch.empty((M, M), device="cuda")
    g = bs.Grid(M, xmax)
    bs.bs_payoff(g, p, u)
    dtau = 1.0 / 4096
    bs.fine_propagate_batched(g, [p], [u], [u], [tau - dtau], [dtau], 1)
    torch.cuda.synchronize()
    got = u.cpu().double().numpy()
    x = np.linspace(0.0, xmax, M)
    for k in range(1, M):
        want = cf.cash_or_nothing(x[k], xmax, 100.0, 100.0, 1.0, r, sigma1, sigma2, rho, tau)
        assert abs(got[M - 1, k] - want) <= TOL, ("y edge", k, got[M - 1, k], want)
        want = cf.cash_or_nothing(xmax, x[k], 100.0, 100.0, 1.0, r, sigma1, sigma2, rho, tau)
        assert abs(got[k, M - 1] - want) <= TOL, ("x edge", k, got[k, M - 1], want)
