"""F on inputs off the 16-byte grid ahead of aligned ones: every copy's source address follows the
state's own alignment, also where the copy only fills zeros outside the domain."""
import pytest

import workloads as wl
from tests.gpu_util import FP32_FINE_TOL, dtau_for, oracle_fine, rel_err, start_state, to_gpu, to_np

pytestmark = pytest.mark.gpu

P = wl.Params(0.3, 0.2, 0.5, 0.05, payoff=wl.BASKET)


# multiples of four, so that aligned states take 16-byte copies: regions wider than the grid (100, 252),
# one vertical region for a grid beyond a cluster's width (260, 288), several regions (300)
@pytest.mark.parametrize("layout", [0, 1, 2])
@pytest.mark.parametrize("M", [100, 252, 260, 288, 300])
def test_unaligned_state_first(M, layout):
    import torch
    import paper_2404_02521_gb300 as bs
    bs.load()
    dtau = dtau_for(M, P)
    u0 = start_state(M, 4.0, P, "payoff", seed=M)
    g = bs.Grid(M, 4.0)
    uin = to_gpu(u0)
    off = torch.empty(M * M + 1, device="cuda")[1:].view(M, M)
    off.copy_(uin)
    bs.bs_set_option(bs.OPT_FINE_TILE, layout)
    try:
        outs = [torch.empty_like(uin) for _ in range(3)]
        bs.fine_propagate_batched(g, [P] * 3, [off, uin, off], outs, [0.05] * 3, [dtau] * 3, 20)
        alone = torch.empty_like(uin)
        bs.fine_propagate_batched(g, [P], [off], [alone], [0.05], [dtau], 20)
        torch.cuda.synchronize()
    finally:
        bs.bs_set_option(bs.OPT_FINE_TILE, 0)
    for out in outs[1:] + [alone]:
        assert torch.equal(outs[0], out)
    assert rel_err(to_np(outs[0]), oracle_fine(M, 4.0, P, u0, 0.05, dtau, 20)) <= FP32_FINE_TOL
