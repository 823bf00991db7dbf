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
