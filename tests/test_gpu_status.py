"""A failure of an asynchronous call is reported by the next synchronous call on the grid, once."""
import pytest

import workloads as wl
from tests.gpu_util import start_state, to_gpu

pytestmark = pytest.mark.gpu


@pytest.fixture(scope="module")
def bs():
    import paper_2404_02521_gb300 as bs
    bs.load()
    yield bs
    bs.bs_set_option(bs.OPT_KRYLOV_MAXIT, 400)
    bs.bs_set_option(bs.OPT_PIPELINE, 1)


# the serial and the pipelined driver; on a grid size whose coarse kernel is measured by an earlier call,
# and by the call that follows the failure (tuning solves have status words of their own)
@pytest.mark.parametrize("pipeline", [0, 1])
@pytest.mark.parametrize("M,tuned", [(48, True), (41, False)])
def test_capped_coarse_step(bs, M, tuned, pipeline):
    import torch
    p = wl.basket_cfg1().params
    pb = wl.Problem("status", M, 4.0, 8, 64, 2, p)
    g, other = bs.Grid(M, 4.0), bs.Grid(M, 4.0)
    u = to_gpu(start_state(M, 4.0, p, "payoff"))
    out = torch.empty_like(u)
    U = torch.empty((pb.N + 1, M, M), device="cuda")

    def solve(grid):
        return bs.parareal_solve(grid, p, pb.N, pb.fine_steps, bs.COARSE_NUM, pb.coarse_steps, None, 1e-4, pb.N, U)

    bs.bs_set_option(bs.OPT_PIPELINE, pipeline)
    if tuned:
        assert solve(other)[0] == 0
    bs.bs_set_option(bs.OPT_KRYLOV_MAXIT, 1)
    bs.coarse_propagate(g, bs.COARSE_NUM, None, p, u, out, 0.0, 0.25, 2)
    bs.bs_set_option(bs.OPT_KRYLOV_MAXIT, 400)
    with pytest.raises(bs.BSError) as e:
        solve(g)
    assert "cap" in str(e.value)
    assert bs.bs_grid_stats(g)[1] is True    # still there to be read, as after any failed solve
    assert solve(g)[0] == 0
    assert bs.bs_grid_stats(g)[1] is False
