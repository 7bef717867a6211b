"""G on grids beyond one cluster (the cooperative grid solver): tile edges, one tile and several per
block, states side by side and one after another, stream capture."""
import pytest

import workloads as wl
from tests.gpu_util import FP32_FINE_TOL, dtau_for, start_state, to_gpu

pytestmark = pytest.mark.gpu

P = wl.Params(0.25, 0.35, 0.7, 0.03, payoff=wl.EXCHANGE)


@pytest.fixture(scope="module")
def bs():
    import paper_2404_02521_gb300 as bs
    bs.load()
    return bs


@pytest.fixture
def tight_g(bs):
    bs.bs_set_option(bs.OPT_KRYLOV_TOL, 1e-6)
    yield
    bs.bs_set_option(bs.OPT_KRYLOV_TOL, 1e-5)


# one node beside a tile's width and height, a full tile grid, and more tiles than resident blocks
@pytest.mark.parametrize("M", [257, 289, 320, 321, 513, 800])
def test_agrees_with_the_jacobi_steps(bs, tight_g, M):
    # both solve the same implicit system: F's first step to 2^-22, G to 1e-6 of the right-hand
    # side; u stays within the fine bound
    import torch
    dtau = dtau_for(M, P, 0.6)
    g = bs.Grid(M, 4.0)
    u = to_gpu(start_state(M, 4.0, P, "payoff"))
    f, c = torch.empty_like(u), torch.empty_like(u)
    bs.fine_propagate_batched(g, [P], [u], [f], [0.1], [dtau], 1)
    bs.coarse_propagate(g, bs.COARSE_NUM, None, P, u, c, 0.1, dtau, 1)
    inplace = u.clone()
    bs.coarse_propagate(g, bs.COARSE_NUM, None, P, inplace, inplace, 0.1, dtau, 1)
    torch.cuda.synchronize()
    assert torch.equal(c, inplace)
    assert float((f - c).abs().max()) <= FP32_FINE_TOL * float(f.abs().max())


@pytest.mark.parametrize("M,B", [(300, 13), (800, 3)])
def test_batched_equals_single(bs, M, B):
    # 300^2 takes 50 blocks a state (several groups, more states than groups); 800^2 all of them
    import torch
    g = bs.Grid(M, 4.0)
    ins = [to_gpu(start_state(M, 4.0, P, "random", seed=b)) for b in range(B)]
    outs = [torch.empty_like(u) for u in ins]
    taus = [0.02 * b for b in range(B)]
    bs.coarse_propagate_batched(g, bs.COARSE_NUM, None, [P] * B, ins, outs, taus, 1.0 / 32, 2)
    one = torch.empty_like(ins[0])
    for b in range(B):
        bs.coarse_propagate(g, bs.COARSE_NUM, None, P, ins[b], one, taus[b], 1.0 / 32, 2)
        torch.cuda.synchronize()
        assert torch.equal(one, outs[b]), b


def test_capture(bs):
    import torch
    M = 300
    g = bs.Grid(M, 4.0)
    u = to_gpu(start_state(M, 4.0, P, "payoff"))
    want, out = torch.empty_like(u), torch.empty_like(u)
    bs.coarse_propagate(g, bs.COARSE_NUM, None, P, u, want, 0.1, 1.0 / 32, 2)
    torch.cuda.synchronize()
    graph = torch.cuda.CUDAGraph()
    with torch.cuda.graph(graph):
        bs.coarse_propagate(g, bs.COARSE_NUM, None, P, u, out, 0.1, 1.0 / 32, 2)
    for _ in range(2):
        out.zero_()
        graph.replay()
        torch.cuda.synchronize()
        assert torch.equal(out, want)


def test_two_streams_at_once(bs):
    # cooperative launches of two grids on two streams, beside F on a third
    import torch
    M = 400
    u = to_gpu(start_state(M, 4.0, P, "payoff"))
    grids = [bs.Grid(M, 4.0) for _ in range(3)]
    streams = [torch.cuda.Stream() for _ in range(3)]
    want = torch.empty_like(u)
    bs.coarse_propagate(grids[0], bs.COARSE_NUM, None, P, u, want, 0.1, 1.0 / 32, 2)
    outs = [torch.empty_like(u) for _ in range(8)]
    f = [torch.empty_like(u) for _ in range(8)]
    torch.cuda.synchronize()
    for k in range(8):
        bs.coarse_propagate(grids[k % 2], bs.COARSE_NUM, None, P, u, outs[k], 0.1, 1.0 / 32, 2, stream=streams[k % 2])
        if k % 4 == 0:
            bs.fine_propagate_batched(grids[2], [P] * 8, [u] * 8, f, [0.1] * 8, [dtau_for(M, P)] * 8, 40,
                                      stream=streams[2])
    torch.cuda.synchronize()
    for g in grids:
        assert bs.bs_grid_stats(g)[1] is False
    for o in outs:
        assert torch.equal(o, want)
