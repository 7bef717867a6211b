"""Register tiles of F at the sizes where their bookkeeping can go wrong: grids one node beside the
tiles' widths and heights, single and overlapping regions, inputs and outputs off the 16-byte
grid, propagations long enough to reuse the far-field ring."""
import numpy as np
import pytest

import workloads as wl
from tests.gpu_util import FP32_FINE_TOL, dtau_for, oracle_fine, rel_err, start_state, to_gpu, to_np

pytestmark = pytest.mark.gpu

PARAMS = {"basket": wl.Params(0.3, 0.2, 0.5, 0.05, payoff=wl.BASKET),
          "exchange": wl.Params(0.25, 0.35, -0.5, 0.03, payoff=wl.EXCHANGE),
          "cash": wl.Params(0.3, 0.25, 0.4, 0.06, payoff=wl.CASH_OR_NOTHING, strike=1.5, strike2=1.4)}


@pytest.fixture(scope="module")
def bs():
    import paper_2404_02521_gb300 as bs
    bs.load()
    yield bs
    bs.bs_set_option(bs.OPT_FINE_TILE, 0)


# widths of 64, 128, 192 and 256 columns, heights of 16 and 32 rows per CTA, one and several
# regions; steps beyond the third far-field chunk of either row count (16 or 8 steps)
@pytest.mark.parametrize("M,payoff,nsteps", [
    (4, "basket", 20), (31, "exchange", 70), (33, "cash", 52), (63, "basket", 70), (65, "exchange", 34),
    (127, "cash", 34), (129, "basket", 34), (191, "exchange", 20), (193, "basket", 20), (255, "cash", 20),
    (257, "exchange", 20), (260, "basket", 20), (333, "cash", 20), (481, "exchange", 18)])
def test_tile_edges(bs, M, payoff, nsteps):
    import torch
    p = PARAMS[payoff]
    dtau = dtau_for(M, p)
    u0 = start_state(M, 4.0, p, "payoff", seed=M)
    g = bs.Grid(M, 4.0)
    uin = to_gpu(u0)
    want = None
    for layout in (1, 2, 0):
        bs.bs_set_option(bs.OPT_FINE_TILE, layout)
        # three states, the last one in and out of buffers off the 16-byte grid
        off_in = torch.empty(M * M + 1, device="cuda")[1:].view(M, M)
        off_in.copy_(uin)
        off_out = torch.empty(M * M + 1, device="cuda")[1:].view(M, M)
        outs = [torch.empty_like(uin), torch.empty_like(uin), off_out]
        bs.fine_propagate_batched(g, [p] * 3, [uin, uin, off_in], outs, [0.05, 0.3, 0.05], [dtau, dtau / 3, dtau],
                                  nsteps)
        torch.cuda.synchronize()
        assert torch.equal(outs[0], outs[2]), layout
        if want is None:
            want = outs
            assert rel_err(to_np(outs[0]), oracle_fine(M, 4.0, p, u0, 0.05, dtau, nsteps)) <= FP32_FINE_TOL
        for a, b in zip(outs, want):
            assert torch.equal(a, b), layout
    bs.bs_set_option(bs.OPT_FINE_TILE, 0)


def test_long_chain_in_pieces_equals_the_steps_one_by_one_in_place(bs):
    # a launch that starts late (all its steps of two sweeps) and a state stepped in place
    import torch
    p, M = PARAMS["basket"], 300
    dtau = dtau_for(M, p)
    u0 = to_gpu(start_state(M, 4.0, p, "payoff", seed=1))
    g = bs.Grid(M, 4.0)
    a, b = torch.empty_like(u0), u0.clone()
    bs.fine_propagate_batched(g, [p], [u0], [a], [0.0], [dtau], 75)
    bs.fine_propagate_batched(g, [p], [b], [b], [0.0], [dtau], 75)
    torch.cuda.synchronize()
    assert torch.equal(a, b)
