"""Far field of the cash-or-nothing option where both strikes lie beyond the grid: values of 1e-13 of the
cash and less, which the correlation makes eleven orders of magnitude larger than the product of the
two one-asset probabilities."""
import numpy as np
import pytest

import workloads as wl
from oracle import fd

pytestmark = pytest.mark.gpu


# The FP32 arguments h and k are within 1e-6 of their values near -7, which moves exp(-h^2 / (1 + rho)) by 1e-5.
@pytest.mark.parametrize("rho", [0.9, 0.5])
def test_both_strikes_beyond_the_grid(rho):
    import torch
    import paper_2404_02521_gb300 as bs
    bs.load()
    p = wl.Params(0.2, 0.2, rho, 0.05, payoff=wl.CASH_OR_NOTHING, strike=1.5, strike2=1.5, cash=1e10)
    M, xmax, tau0, dtau = 33, 1.0, 0.08, 0.01
    g = bs.Grid(M, xmax)
    u = torch.zeros((M, M), device="cuda")
    out = torch.empty_like(u)
    bs.fine_propagate_batched(g, [p], [u], [out], [tau0], [dtau], 1)
    torch.cuda.synchronize()
    X, Y = fd.mesh(M, xmax)
    want = fd.dirichlet(p)(X, Y, tau0 + dtau)
    for got, edge in ((out[M - 1], want[M - 1]), (out[:, M - 1], want[:, M - 1])):
        got = got.cpu().double().numpy()
        assert np.max(np.abs(got - edge)) <= 1e-4 * np.max(edge), (got[-3:], edge[-3:])
