"""The forms of the fused step (marching, tiles of 24 rows and of 16, 14 and 12;
block_x 64, 128, 256) at the sizes where they can go wrong: one column or row short
of, at and past a strip, a pair of strips and a tile, domains narrower than a
strip, and segments that a block walks tile by tile. Every form gives the same
bits, heat flux included, and one step agrees with the FP64 oracle within the
one-step bound of test_gpu_parity.py (a few ulp per operation, 2e-6)."""

import numpy as np
import pytest
import torch

from paper_1501_03857_gb300 import inputs
from parity_util import norm_err, oracle_params, run_oracle, theta_err

pytestmark = pytest.mark.gpu

FORMS = ((64, 0), (128, 0), (256, 0), (256, 2), (256, 3), (64, 1), (64, 9), (128, 5), (128, 40), (256, 17))
# (Lx, Ly, bc, ghost, isothermal)
CASES = [(53, 5, 0, False, False), (54, 6, 1, False, False), (55, 7, 0, True, False), (107, 13, 0, False, False),
         (108, 14, 2, False, False), (109, 15, 1, True, False), (3, 27, 0, False, False), (64, 28, 2, False, True),
         (163, 29, 0, False, True), (31, 3, 0, False, False), (33, 12, 1, False, False), (60, 4, 2, False, False)]


@pytest.mark.parametrize("Lx,Ly,bc,ghost,iso", CASES)
def test_forms_agree_and_match_the_oracle(Lx, Ly, bc, ghost, iso):
    assert torch.cuda.is_available(), "GPU tests need CUDA"
    from paper_1501_03857_gb300 import lb
    cfg = lb.Config(Lx=Lx, Ly=Ly, bc_y=bc, ghost_layer=ghost, isothermal=iso)
    rv, rl = lb.coexistence(cfg)
    rho0, f0, th0 = inputs.random_state(Lx, Ly, rl, rv, Ly * 0.45, seed=Lx + 1000 * Ly)
    ref = None
    for form in FORMS:
        sim = lb.Simulation(cfg, superheat=0.012, Gw=0.05, rho0=rho0)
        sim.set_launch(*form)
        sim.set_state(f0, th0)
        sim.step(1)
        one = sim.get_state() + (sim.heat_flux(),)
        sim.step(36)  # a captured run of 32 steps and single ones
        got = one + sim.get_state() + (sim.heat_flux(),)
        sim.close()
        if ref is None:
            ref = got
            continue
        for a, b in zip(got, ref):
            assert a == b if isinstance(a, dict) else np.array_equal(a, b), form
    P = oracle_params(cfg, rho0, superheat=0.012, Gw=0.05)
    fr, tr, qs = run_oracle(f0, th0, P, 1)
    assert norm_err(ref[0], fr.numpy()) < 2e-6
    assert theta_err(ref[1], tr.numpy(), 0.012) < 2e-6
    if bc != 2:
        assert ref[2]["n"] == 1 and abs(ref[2]["q_inst"] - qs[0]) <= 1e-5 * abs(qs[0]) + 1e-12
        assert ref[5]["n"] == 37
