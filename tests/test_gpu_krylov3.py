"""Three-asset G as one cooperative launch: sizes with one tile and several per block, the iteration
cap."""
import types

import pytest

import workloads as wl
from tests.gpu_util import FP32_FINE_TOL

pytestmark = pytest.mark.gpu


@pytest.fixture(scope="module")
def bs():
    import paper_2404_02521_gb300 as bs
    bs.load()
    return bs


def option(payoff, strike=1.0):
    return types.SimpleNamespace(sigma=(0.3, 0.2, 0.25), rho=(0.5, -0.3, 0.2), r=0.05, strike=strike,
                                 w=(0.4, 0.35, 0.25), payoff=payoff)


# 4 and 5 nodes: a part of one tile; 32 to 34: a tile's width and one node beside it; 128: more
# tiles than blocks
@pytest.mark.parametrize("M", [4, 5, 32, 33, 34, 65, 128])
@pytest.mark.parametrize("payoff", [wl.BASKET, wl.EXCHANGE])
def test_coarse3_agrees_with_the_jacobi_steps(bs, M, payoff):
    # both solve the same implicit system: F's first step to 2^-22, G to 1e-6 of the
    # right-hand side; u stays within the fine bound plus 1e-6 of the increment
    import torch
    p, dtau = option(payoff), 2.0 / M ** 2
    u = torch.empty((M, M, M), device="cuda")
    bs.bs_payoff3(M, 4.0, p, u)
    f, g = torch.empty_like(u), torch.empty_like(u)
    bs.bs_set_option(bs.OPT_KRYLOV_TOL, 1e-6)
    try:
        bs.fine_propagate3(M, 4.0, p, [u], [f], [0.1], dtau, 1)
        bs.coarse_propagate3(M, 4.0, p, u, g, 0.1, dtau, 1)
        inplace = u.clone()
        bs.coarse_propagate3(M, 4.0, p, inplace, inplace, 0.1, dtau, 1)
    finally:
        bs.bs_set_option(bs.OPT_KRYLOV_TOL, 1e-5)
    torch.cuda.synchronize()
    assert torch.equal(g, inplace)
    assert float((f - g).abs().max()) <= FP32_FINE_TOL * float(f.abs().max())


def test_coarse3_iteration_cap(bs):
    import torch
    p, M = option(wl.BASKET), 24
    u = torch.empty((M, M, M), device="cuda")
    bs.bs_payoff3(M, 4.0, p, u)
    out, want = torch.full_like(u, 7.0), torch.empty_like(u)
    bs.coarse_propagate3(M, 4.0, p, u, want, 0.0, 0.2, 2)
    bs.bs_set_option(bs.OPT_KRYLOV_MAXIT, 1)
    try:
        with pytest.raises(bs.BSError):
            bs.coarse_propagate3(M, 4.0, p, u, out, 0.0, 0.2, 2)
        U = torch.empty((5, M, M, M), device="cuda")
        with pytest.raises(bs.BSError):
            bs.parareal_solve3(M, 4.0, p, 0.8, 4, 80, 2, 1e-4, 4, U)
    finally:
        bs.bs_set_option(bs.OPT_KRYLOV_MAXIT, 400)
    torch.cuda.synchronize()
    assert bool((out == 7.0).all())
    bs.coarse_propagate3(M, 4.0, p, u, out, 0.0, 0.2, 2)
    torch.cuda.synchronize()
    assert torch.equal(out, want)
