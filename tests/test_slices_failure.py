"""A rank whose kernels failed ends the partitioned Parareal on every rank after the same iteration (CPU
ranks on the gloo backend; the failure is the backend's own word for it)."""
import os

import pytest

import workloads as wl
from paper_2404_02521_gb300.slices import parareal_partitioned
from tests.test_slices_gloo import OracleSlices, _free_port


class FailingSlices(OracleSlices):
    """The second rank's work fails in the second iteration."""

    def __init__(self, pb, rank, bits):
        super().__init__(pb)
        self.rank, self.bits, self.asked = rank, bits, 0

    def failure(self):
        self.asked += 1
        return self.bits if self.rank == 1 and self.asked == 2 else 0


def _worker(rank, world, port, pb, bits, out):
    import torch.distributed as dist
    os.environ["MASTER_ADDR"] = "127.0.0.1"
    os.environ["MASTER_PORT"] = str(port)
    dist.init_process_group("gloo", rank=rank, world_size=world)
    be = FailingSlices(pb, rank, bits)
    try:
        parareal_partitioned(be, pb.N, 0.0, pb.N)
        out[rank] = ("solved", be.asked)
    except RuntimeError as e:
        out[rank] = (str(e), be.asked)
    dist.barrier()
    dist.destroy_process_group()


@pytest.mark.parametrize("bits,word", [(1, "iteration cap"), (2, "timed out"), (3, "timed out")])
def test_every_rank_raises(bits, word):
    import torch.multiprocessing as mp
    pb = wl.Problem("slices", 14, 4.0, 6, 12, 1, wl.exchange_cfg2(0.7).params)
    with mp.Manager() as m:
        out = m.dict()
        mp.spawn(_worker, args=(2, _free_port(), pb, bits, out), nprocs=2, join=True)
        res = dict(out)
    for rank in range(2):
        assert word in res[rank][0] and res[rank][1] == 2, res
