"""Device-to-device state copies (lb_set_state / lb_get_state with on_device):
widths with and without 16-byte rows, rows longer than one warp's run, buffers
that start off a 16-byte boundary, either part alone, and memory that is not
this device's (the copies then go through the runtime); all bytes arrive and
nothing beside them is written. Batch statistics read in one launch equal the
instances' own."""

import numpy as np
import pytest
import torch

pytestmark = pytest.mark.gpu


@pytest.fixture(scope="module")
def lb():
    assert torch.cuda.is_available(), "GPU tests need CUDA"
    from paper_1501_03857_gb300 import lb as lbmod
    return lbmod


@pytest.mark.parametrize("Lx,Ly", [(1, 3), (36, 5), (37, 4), (1024, 3), (1028, 3), (2051, 3)])
@pytest.mark.parametrize("off", [0, 1])
def test_device_state_round_trip(lb, Lx, Ly, off):
    sim = lb.Simulation(lb.Config(Lx=Lx, Ly=Ly, bc_y=lb.BC_PERIODIC))
    n = Lx * Ly
    g = torch.Generator().manual_seed(Lx)
    f, t = torch.rand(9 * n, generator=g) + 0.5, torch.rand(n, generator=g)
    fd, td = torch.zeros(9 * n + 8, device="cuda"), torch.zeros(n + 8, device="cuda")
    fd[off:off + 9 * n], td[off:off + n] = f.cuda(), t.cuda()
    ptr = lambda x: x.data_ptr() + 4 * off
    lb.check(lb.lib.lb_set_state(sim.h, ptr(fd), None, 1))
    lb.check(lb.lib.lb_set_state(sim.h, None, ptr(td), 1))
    hf, ht = sim.get_state()
    assert np.array_equal(hf.ravel(), f.numpy()) and np.array_equal(ht.ravel(), t.numpy())
    fo, to = torch.full((9 * n + 8,), -1.0, device="cuda"), torch.full((n + 8,), -1.0, device="cuda")
    lb.check(lb.lib.lb_get_state(sim.h, ptr(fo), ptr(to), 1))
    for o, v, m in ((fo, f, 9 * n), (to, t, n)):
        o = o.cpu()
        assert torch.equal(o[off:off + m], v) and bool((o[:off] == -1).all()) and bool((o[off + m:] == -1).all())
    pinned = torch.zeros(9 * n).pin_memory()
    lb.check(lb.lib.lb_get_state(sim.h, pinned.data_ptr(), None, 1))
    assert torch.equal(pinned, f)
    sim.close()


def test_batch_statistics_equal_the_instances(lb):
    cfgs = [lb.Config(Lx=40 + 9 * i, Ly=24, pool_height=10.0, seed=i) for i in range(3)]
    batch = lb.Batch([{"cfg": c, "superheat": 0.01 + 0.002 * i} for i, c in enumerate(cfgs)])
    batch.step(5)
    first = batch.heat_flux(reset=True)
    again = batch.heat_flux()
    batch.step(3)
    last = batch.heat_flux()
    for i, c in enumerate(cfgs):
        sim = lb.Simulation(c, superheat=0.01 + 0.002 * i)
        sim.step(5)
        a = sim.heat_flux(reset=True)
        sim.step(3)
        b = sim.heat_flux()
        sim.close()
        for k in ("q_inst", "q_mean", "q_std", "n"):
            assert first[k][i] == a[k] and last[k][i] == b[k], (i, k)
        assert again["n"][i] == 0 and again["q_inst"][i] == a["q_inst"]
    batch.close()
