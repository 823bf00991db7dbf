"""The launch shape that info() reports is one that set_launch() takes, and
chooses the same shape again: for the automatic choice over domains that take
each form, for every form asked for, and for batches (per step and
persistent)."""

import pytest
import torch

pytestmark = pytest.mark.gpu


@pytest.fixture(scope="module")
def lb():
    assert torch.cuda.is_available(), "GPU tests need CUDA"
    from paper_1501_03857_gb300 import lb as lbmod
    return lbmod


@pytest.mark.parametrize("Lx,Ly", [(1, 3), (100, 100), (300, 100), (600, 150), (517, 1003), (2048, 700), (5000, 7),
                                   (20000, 5)])
def test_simulation_shape_round_trip(lb, Lx, Ly):
    sim = lb.Simulation(lb.Config(Lx=Lx, Ly=Ly, pool_height=0.4 * Ly))
    for asked in ((0, 0), (64, 0), (128, 0), (256, 0), (64, 9), (128, 5), (256, 2), (256, 4), (256, 17), (0, 12)):
        sim.set_launch(*asked)
        info = sim.info()
        assert info["block_x"] in (64, 128, 256) and asked[0] in (0, info["block_x"])
        sim.set_launch(info["block_x"], info["seg_rows"])
        assert sim.info() == info, asked
    sim.close()


@pytest.mark.parametrize("n,Lx,Ly", [(3, 40, 24), (36, 600, 150)])
@pytest.mark.parametrize("tpb", [0, 1])
def test_batch_shape_round_trip(lb, n, Lx, Ly, tpb):
    batch = lb.Batch([{"cfg": lb.Config(Lx=Lx, Ly=Ly, pool_height=0.4 * Ly, seed=i), "superheat": 0.01} for i in range(n)])
    batch.set_persistent(tpb)
    for block_x in (128, 64):
        batch.set_launch(block_x, 0)
        info = batch.info()
        assert info["block_x"] == block_x
        batch.set_launch(info["block_x"], 0)
        assert batch.info() == info
    batch.close()
