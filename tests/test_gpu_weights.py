"""Kernel weights of the double plans: the polynomial of the default kernel
shape and the definition a caller's own shape falls back to, against the FP64
oracle through Phi, Phi^dagger and the normal operator."""
import numpy as np
import pytest
import torch

import paper_1502_05037_gb300 as pk
from gpu_util import DEV, TOL, rel
from oracle import nufft as onf
from paper_1502_05037_gb300 import synth

pytestmark = pytest.mark.gpu


@pytest.mark.parametrize("J", [2, 3, 4, 5, 6, 7, 8])
@pytest.mark.parametrize("shape", [0.0, 5.0])
def test_double_weights(J, shape):
    nx, ny, M = 32, 16, 701
    u, v = synth.uv_coverage(M, 2000 + J, uniform_fraction=0.3)
    op = onf.NufftPlan(nx, ny, u, v, J, beta=shape * J if shape else None)
    plan = pk.Plan(nx, ny, torch.from_numpy(u).to(DEV), torch.from_numpy(v).to(DEV), kb_width=J, levels=2,
                   kb_beta=shape * J, dtype=pk.PURIFY_F64)
    g = synth.rng(J)
    x = g.standard_normal((ny, nx))
    y = g.standard_normal(M) + 1j * g.standard_normal(M)
    xd, yd = torch.from_numpy(x).to(DEV), torch.from_numpy(y).to(DEV)
    got_y = torch.empty(M, dtype=torch.complex128, device=DEV)
    got_x = torch.empty((ny, nx), dtype=torch.complex128, device=DEV)
    got_n = torch.empty((ny, nx), dtype=torch.float64, device=DEV)
    pk.purify_phi(plan, xd, got_y)
    pk.purify_phi_adj(plan, yd, got_x)
    pk.purify_phi_normal(plan, xd, got_n)
    tol = TOL[pk.PURIFY_F64]
    assert rel(got_y.cpu(), onf.phi(op, x)) <= tol
    assert rel(got_x.cpu(), onf.phi_adj(op, y)) <= tol
    assert rel(got_n.cpu(), np.real(onf.phi_adj(op, onf.phi(op, x)))) <= tol
