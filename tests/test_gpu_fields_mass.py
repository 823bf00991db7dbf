"""lb_fields in one pass and the mass sum at the sizes where they can go
wrong: columns at the edges of a block's 126 and of the mass sum's runs,
rows at the edges of a segment's 16, every boundary treatment. The fields
agree with lb_fields_noalloc (the same formulas through scratch planes) to the
rounding of a few operations; the mass is the exact sum up to the FP64 sum of
runs, also with values far outside the range whose sums need no rounding."""

import math

import numpy as np
import pytest
import torch

from paper_1501_03857_gb300 import inputs

pytestmark = pytest.mark.gpu

SIZES = [(1, 3, 0, False), (125, 15, 0, False), (126, 16, 1, True), (127, 17, 2, False), (253, 33, 0, True),
         (600, 31, 1, False), (129, 32, 2, False)]


@pytest.fixture(scope="module")
def lb():
    assert torch.cuda.is_available(), "GPU tests need CUDA"
    from paper_1501_03857_gb300 import lb as lbmod
    return lbmod


@pytest.mark.parametrize("Lx,Ly,bc,ghost", SIZES)
def test_fields_agree_with_the_two_pass_form(lb, Lx, Ly, bc, ghost):
    cfg = lb.Config(Lx=Lx, Ly=Ly, bc_y=bc, ghost_layer=ghost)
    rv, rl = lb.coexistence(cfg)
    rho0, f0, th0 = inputs.random_state(Lx, Ly, rl, rv, Ly * 0.45, seed=Lx + Ly)
    sim = lb.Simulation(cfg, superheat=0.01, Gw=0.08, rho0=rho0)
    sim.set_state(f0, th0)
    got = sim.fields()
    dev = [torch.empty(Ly, Lx, device="cuda") for _ in range(4)]
    sim.fields_device(*dev)
    ref = [torch.empty(Ly, Lx, device="cuda") for _ in range(4)]
    lb.fields_noalloc(cfg, 0.08, float(np.asarray(rho0, np.float64).mean()), torch.from_numpy(f0).cuda(),
                      torch.from_numpy(th0).cuda(), *ref)
    speed = float(torch.hypot(ref[1], ref[2]).max())
    for k, d, r, scale in zip(("rho", "ux", "uy", "T"), dev, ref, (float(ref[0].max()), speed, speed, 1.0)):
        assert np.array_equal(got[k], d.cpu().numpy()), k
        # u: psi's few-ulp differences amplified by |F| / (rho |v|), as against the oracle
        assert float((d - r).abs().max()) <= 1e-5 * scale, k
    sim.close()


@pytest.mark.parametrize("Lx,Ly", [(1, 3), (37, 9), (128, 5), (2047, 4), (2050, 3), (4100, 3)])
@pytest.mark.parametrize("lo,hi", [(-4, 2), (-30, -18), (5, 14), (-25, 12)])
def test_mass_is_the_exact_sum(lb, Lx, Ly, lo, hi):
    """Values 2^lo .. 2^hi of both signs; the bound is the FP64 rounding of a
    sum of at most 9 Lx Ly terms in any order, n 2^-53 of the sum of |f|."""
    cfg = lb.Config(Lx=Lx, Ly=Ly, bc_y=lb.BC_PERIODIC)
    sim = lb.Simulation(cfg)
    n = 9 * Lx * Ly
    rng = np.random.default_rng(Lx + Ly)
    f = (2.0 ** rng.uniform(lo, hi, n) * np.where(rng.random(n) < 0.3, -1.0, 1.0)).astype(np.float32)
    sim.set_state(f.reshape(9, Ly, Lx), None)
    exact = math.fsum(f.astype(np.float64))
    assert abs(sim.mass() - exact) <= n * 2.0 ** -53 * float(np.abs(f.astype(np.float64)).sum())
    sim.close()
