"""The adjoint's two forms against the FP64 oracle's autograd adjoint: the
tiled reverse step at the sizes where its tiles change (24 rows in one tile;
18 + 12 k + 18 rows after that, a last tile that would hold one row; 52
columns a strip), over windows long enough for the second tile to matter, and
the marching reverse kernels on a domain too large for the tiles. Bound: a
few FP32 ulp per reverse step through tens of steps, 1e-4."""

import numpy as np
import pytest
import torch

from test_gpu_adjoint import F64, gpu_adjoint, lb, oracle_J, rel, setup  # noqa: F401

pytestmark = pytest.mark.gpu


@pytest.mark.parametrize("Lx,Ly,outflow,ghost,n", [(52, 24, False, False, 30), (53, 25, True, False, 40),
                                                   (105, 36, False, True, 40), (20, 37, True, False, 50),
                                                   (31, 49, False, False, 50), (1250, 230, True, False, 3)])
def test_reverse_forms_match_oracle_autograd(lb, Lx, Ly, outflow, ghost, n):  # noqa: F811
    cfg, rho0, prof, P, f0, th0 = setup(lb, Lx=Lx, Ly=Ly, bc=lb.BC_TOP_OUTFLOW if outflow else None, ghost=ghost)
    tb = torch.tensor(prof, dtype=F64, requires_grad=True)
    gw = torch.tensor(0.05, dtype=F64, requires_grad=True)
    Jo = oracle_J(P, f0, th0, tb, gw, n)
    gtb, ggw = torch.autograd.grad(Jo, (tb, gw))
    J, dTb, dGw = gpu_adjoint(lb, cfg, rho0, prof, 0.05, f0, th0, n, ckpt=1)
    print(f"{Lx}x{Ly}: J {abs(J / float(Jo.detach()) - 1):.1e} dTb {rel(dTb, gtb.numpy()):.1e} "
          f"dGw {abs(dGw / float(ggw) - 1):.1e}")
    assert abs(J / float(Jo.detach()) - 1) < 1e-5
    assert rel(dTb, gtb.numpy()) < 1e-4
    assert abs(dGw / float(ggw) - 1) < 1e-4


@pytest.mark.parametrize("Ly,outflow,ghost", [(3, False, False), (3, True, False), (4, False, True), (5, True, False),
                                              (8, False, False), (9, True, True), (17, False, False), (30, True, False),
                                              (31, False, True)])
def test_marching_reverse_on_wide_low_domains(lb, Ly, outflow, ghost):  # noqa: F811
    """The marching reverse kernels (too many strips for the tiles) where their
    segments are a few rows, end on an odd row or hold no steady iteration.
    Three steps of a few hundred FP32 operations each: 1e-5 of each column's
    share, in the norm and at the worst column; dJ/dG_w is the sum of 23773
    shares of both signs (their magnitudes come to 45 times the sum at 31
    rows), so its bound is 1e-5 of the sum of magnitudes."""
    Lx = 23773
    cfg, rho0, prof, P, f0, th0 = setup(lb, Lx=Lx, Ly=Ly, bc=lb.BC_TOP_OUTFLOW if outflow else None, ghost=ghost)
    tb = torch.tensor(prof, dtype=F64, requires_grad=True)
    gw = torch.full((Lx,), 0.05, dtype=F64, requires_grad=True)  # one per column
    Jo = oracle_J(P, f0, th0, tb, gw, 3)
    gtb, ggw = torch.autograd.grad(Jo, (tb, gw))
    J, dTb, dGw = gpu_adjoint(lb, cfg, rho0, prof, 0.05, f0, th0, 3, ckpt=1)
    worst = float(np.abs(dTb - gtb.numpy()).max() / np.abs(gtb.numpy()).max())
    print(f"{Lx}x{Ly}: J {abs(J / float(Jo.detach()) - 1):.1e} dTb {rel(dTb, gtb.numpy()):.1e} worst {worst:.1e} "
          f"dGw {abs(dGw - float(ggw.sum())) / float(ggw.abs().sum()):.1e}")
    assert abs(J / float(Jo.detach()) - 1) < 1e-5
    assert rel(dTb, gtb.numpy()) < 1e-5 and worst < 1e-5
    assert abs(dGw - float(ggw.sum())) < 1e-5 * float(ggw.abs().sum())
