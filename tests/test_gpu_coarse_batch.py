"""G on several states beyond one cluster: a state's result is the same bit for bit alone and in a batch,
however many blocks and rounds of groups the batch gets."""
import pytest

import workloads as wl
from tests.gpu_util import start_state, to_gpu

pytestmark = pytest.mark.gpu

P = wl.Params(0.25, 0.35, 0.7, 0.03, payoff=wl.EXCHANGE)


# a tile per block in one or several groups (300, 512); more than half of the resident blocks per state
# (513 and 577: 153 and 190 tiles), alone in registers, in a batch through the workspace; more tiles than
# resident blocks (800), and more than three per SM (1000), one state or two in a group of blocks; groups
# that come round a second time
@pytest.mark.parametrize("M,B", [(300, 8), (512, 2), (512, 7), (513, 2), (513, 5), (513, 9), (577, 3), (577, 7), (800, 2),
                                 (1000, 2)])
def test_alone_and_in_a_batch(M, B):
    import torch
    import paper_2404_02521_gb300 as bs
    bs.load()
    g = bs.Grid(M, 4.0)
    ins = [to_gpu(start_state(M, 4.0, P, "random", seed=b)) for b in range(B)]
    outs = [torch.empty_like(u) for u in ins]
    taus = [0.02 * b for b in range(B)]
    bs.coarse_propagate_batched(g, bs.COARSE_NUM, None, [P] * B, ins, outs, taus, 1.0 / 32, 2)
    one = torch.empty_like(ins[0])
    for b in sorted({0, B // 2, B - 1}):
        bs.coarse_propagate(g, bs.COARSE_NUM, None, P, ins[b], one, taus[b], 1.0 / 32, 2)
        torch.cuda.synchronize()
        assert torch.equal(one, outs[b]), b
    assert bs.bs_grid_stats(g)[1] is False
