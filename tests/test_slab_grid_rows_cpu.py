"""Every rank of a decomposed grid learns the whole grid's rows before its first
step (slab.RankSlab.init): gloo ranks around a stand-in band."""
import os
import socket

import pytest
import torch
import torch.distributed as dist
import torch.multiprocessing as mp

HEIGHTS = [16, 8, 13]


class FakeBand:
    device = "cpu"

    def __init__(self, rank):
        self.Ny, self.calls = HEIGHTS[rank], []

    def set_grid_rows(self, rows):
        self.calls.append(("rows", rows))

    def init(self, *fields):
        self.calls.append(("init", len(fields)))

    def halo_pack(self, lo, hi):
        pass

    def halo_unpack(self, lo, hi):
        pass


def _worker(rank, world, port, out):
    from paper_2510_04197_gb300 import slab
    os.environ["MASTER_ADDR"], os.environ["MASTER_PORT"] = "127.0.0.1", str(port)
    dist.init_process_group("gloo", rank=rank, world_size=world)
    try:
        rs = object.__new__(slab.RankSlab)  # a band without the library
        rs.dist, rs.rank, rs.world, rs.periodic, rs.fixed_dt = dist, rank, world, True, True
        rs.sim = FakeBand(rank)
        rs.send_lo, rs.send_hi, rs.recv_lo, rs.recv_hi = (torch.zeros(2) for _ in range(4))
        rs.init(0, 0, 0, 0)
        torch.save(rs.sim.calls, f"{out}.{rank}")
    finally:
        dist.destroy_process_group()


@pytest.mark.parametrize("world", [2, 3])
def test_rows_are_summed_over_the_ranks(tmp_path, world):
    s = socket.socket()
    s.bind(("127.0.0.1", 0))
    port = s.getsockname()[1]
    s.close()
    out = str(tmp_path / "rows")
    mp.start_processes(_worker, args=(world, port, out), nprocs=world, join=True, start_method="spawn")
    for r in range(world):
        assert torch.load(f"{out}.{r}") == [("rows", sum(HEIGHTS[:world])), ("init", 4)]
