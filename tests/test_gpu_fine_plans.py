"""One long propagation under launch plans that cut it into different launches, against the oracle: the
pieces of the cold first step, the early steps, and launches that hold late steps alone."""
import pytest

import workloads as wl
from tests.gpu_util import FP32_FINE_TOL, dtau_for, oracle_fine, rel_err, start_state, to_gpu, to_np

pytestmark = pytest.mark.gpu

P = wl.Params(0.3, 0.2, 0.5, 0.05, payoff=wl.BASKET)


# several regions: the layouts' overlaps allow launches of different length.  300 and 301 take 16-byte and
# 4-byte copies
@pytest.mark.parametrize("M", [300, 301])
def test_plans_agree_with_the_oracle(M):
    import torch
    import paper_2404_02521_gb300 as bs
    bs.load()
    dtau, steps = dtau_for(M, P), 75
    u0 = start_state(M, 4.0, P, "payoff", seed=1)
    want = oracle_fine(M, 4.0, P, u0, 0.0, dtau, steps)
    g, first = bs.Grid(M, 4.0), None
    try:
        for layout in (0, 1, 2):
            bs.bs_set_option(bs.OPT_FINE_TILE, layout)
            out, inplace = torch.empty((M, M), device="cuda"), to_gpu(u0)
            bs.fine_propagate_batched(g, [P], [to_gpu(u0)], [out], [0.0], [dtau], steps)
            bs.fine_propagate_batched(g, [P], [inplace], [inplace], [0.0], [dtau], steps)
            torch.cuda.synchronize()
            first = out if first is None else first
            assert torch.equal(out, first) and torch.equal(inplace, first), layout
    finally:
        bs.bs_set_option(bs.OPT_FINE_TILE, 0)
    assert rel_err(to_np(first), want) <= FP32_FINE_TOL
