"""The marching reverse kernels of the adjoint (rev_thermal_fused,
rev_flow_fused), which take over where a domain has more tiles than the GPU has
SMs: in the checked build they flag no address and give the gradients of the
normal build within rounding (1e-6 relative, as test_gpu_checked.py bounds the
adjoints), for walls, the outflow top and the ghost layer, segments that are
replayed and every step stored. In the normal build both modes give the same
bits: the replayed steps are the stored ones, and the reverse kernels are the
same."""

import os
import subprocess
import sys

import numpy as np
import pytest
import torch

pytestmark = pytest.mark.gpu

ROOT = os.path.dirname(os.path.dirname(os.path.abspath(__file__)))
if ROOT not in sys.path:  # run as a script below
    sys.path.insert(0, ROOT)

# (Lx, Ly, bc, ghost, steps): three rows over many strips; odd sizes; segments
# of four rows with a top row joined to the one below; a deep domain
CASES = [(8003, 3, 0, 0, 4), (8003, 4, 1, 0, 4), (4151, 25, 0, 1, 5), (1873, 61, 1, 1, 5), (1250, 230, 1, 0, 5),
         (1301, 131, 0, 0, 5), (517, 900, 0, 0, 3)]


def tiles(Lx, Ly):
    """Tiles of the tiled reverse step: 52 columns; 24 rows in one, else 18 at
    either end and 12 between."""
    rows = 1 if Ly <= 24 else 2 + max(0, -(-(Ly - 36) // 12))
    return -(-Lx // 52) * rows


def gradients(case, ckpt):
    from paper_1501_03857_gb300 import inputs, lb
    Lx, Ly, bc, ghost, n = case
    cfg = lb.Config(Lx=Lx, Ly=Ly, bc_y=bc, pool_height=0.45 * Ly, ghost_layer=bool(ghost))
    rv, rl = lb.coexistence(cfg)
    rho0 = inputs.pool_density(Lx, Ly, rl, rv, 0.45 * Ly, noise_amp=1e-2, seed=Lx + 7 * Ly)
    sim = lb.Simulation(cfg, superheat=0.012, Gw=0.05, rho0=rho0)
    J, dTb, dGw = sim.adjoint(n, ckpt)
    sim.close()
    return np.concatenate([[J, dGw], dTb])


def test_cases_reach_the_marching_kernels():
    sms = torch.cuda.get_device_properties(0).multi_processor_count
    assert all(tiles(*c[:2]) > sms for c in CASES)


def run(lib, tmp_path):
    out = os.path.join(str(tmp_path), lib + ".npz")
    env = dict(os.environ, PYTHONPATH=ROOT, LBBOIL_LIB=os.path.join(ROOT, "paper_1501_03857_gb300", "_lib", lib))
    r = subprocess.run([sys.executable, os.path.abspath(__file__), out], env=env, capture_output=True, text=True,
                       timeout=600)
    assert r.returncode == 0, r.stdout + r.stderr
    return np.load(out)


def test_checked_build_agrees_and_modes_equal(tmp_path):
    assert torch.cuda.is_available(), "GPU tests need CUDA"
    checked, normal = run("liblbboil_checked.so", tmp_path), run("liblbboil.so", tmp_path)
    worst = 0.0
    for k, case in enumerate(CASES):
        assert np.isfinite(normal[f"{k}_1"]).all()
        assert np.array_equal(normal[f"{k}_1"], normal[f"{k}_2"]), case  # every step stored, replayed
        for mode in (1, 2):
            a, b = checked[f"{k}_{mode}"], normal[f"{k}_{mode}"]
            # J; dJ/dG_w and dJ/dT_b against their largest entry (columns' shares of both signs)
            err = max(abs(a[0] / b[0] - 1), abs(a[1] - b[1]) / abs(b[1]), np.abs(a[2:] - b[2:]).max() / np.abs(b[2:]).max())
            worst = max(worst, float(err))
            assert err < 1e-6, (case, mode, err)
    print(f"largest relative difference: {worst:.1e}")


if __name__ == "__main__":
    np.savez(sys.argv[1], **{f"{k}_{mode}": gradients(c, mode) for k, c in enumerate(CASES) for mode in (1, 2)})
