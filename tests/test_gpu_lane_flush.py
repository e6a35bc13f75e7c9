"""G^H by lanes with every lane adding its own patch rows and with a set's
patches added in common, on either side of the rule between them (kernel width
and grid size), and the lanes' staging at every width - against the FP64
oracle."""
import numpy as np
import pytest
import torch

import paper_1502_05037_gb300 as pk
from gpu_util import DEV, TOL, np_cplx, rel
from oracle import nufft as onf
from paper_1502_05037_gb300 import synth

pytestmark = pytest.mark.gpu


@pytest.mark.parametrize("mode", [3, 4, 5, 6])
@pytest.mark.parametrize("J", [2, 3, 4, 5, 6])
@pytest.mark.parametrize("nx,ny,M", [(16, 32, 3001), (512, 512, 20001)])
def test_lanes_of_the_whole_plane(nx, ny, M, J, mode):
    u, v = synth.uv_coverage(M, 40 + J, uniform_fraction=0.2, dtype=np.float32)
    op = onf.NufftPlan(nx, ny, u.astype(np.float64), v.astype(np.float64), J)
    plan = pk.Plan(nx, ny, torch.from_numpy(u).to(DEV), torch.from_numpy(v).to(DEV), kb_width=J, levels=2,
                   grid_mode=mode)
    g = synth.rng(J + mode)
    x = g.standard_normal((ny, nx)).astype(np.float32)
    y = (g.standard_normal(M) + 1j * g.standard_normal(M)).astype(np.complex64)
    xd, yd = torch.from_numpy(x).to(DEV), torch.from_numpy(y).to(DEV)
    got_y, got_a, got_n = torch.empty_like(yd), torch.empty((ny, nx), dtype=torch.complex64, device=DEV), torch.empty_like(xd)
    pk.purify_phi(plan, xd, got_y)
    pk.purify_phi_adj(plan, yd, got_a)
    pk.purify_phi_normal(plan, xd, got_n)
    want = onf.phi(op, x.astype(np.float64))
    tol = TOL[pk.PURIFY_F32]
    assert rel(got_y.cpu(), want) <= tol
    assert rel(got_a.cpu(), onf.phi_adj(op, y.astype(np.complex128))) <= tol
    assert rel(got_n.cpu(), np.real(onf.phi_adj(op, want))) <= tol


@pytest.mark.parametrize("nx,ny,M,J", [(128, 128, 2001, 6), (512, 512, 20001, 6), (512, 512, 20001, 5),
                                       (1024, 1024, 20001, 5), (256, 256, 20001, 7), (128, 128, 2001, 8),
                                       (512, 512, 20001, 4), (256, 128, 20001, 8)])
def test_solver_adjoint_on_the_half_plane(nx, ny, M, J):
    """The first primal-dual step from x = 0 (and dual variables 0) is the
    solver's adjoint of the projected data; compared with tile subproblems on the
    whole plane, which no rule here touches."""
    u, v = synth.uv_coverage(M, 50 + J, uniform_fraction=0.2, dtype=np.float32)
    ud, vd = torch.from_numpy(u).to(DEV), torch.from_numpy(v).to(DEV)
    g = synth.rng(J)
    y = torch.from_numpy((g.standard_normal(M) + 1j * g.standard_normal(M)).astype(np_cplx(pk.PURIFY_F32))).to(DEV)
    out = []
    for kw in (dict(tile=16), dict(grid_mode=1)):
        plan = pk.Plan(nx, ny, ud, vd, kb_width=J, levels=2, **kw)
        assert plan.info.degrid_mode == (8 if "tile" in kw else 1)
        x = torch.zeros((ny, nx), dtype=torch.float32, device=DEV)
        pk.purify_pd_solve(plan, y, np.array([1e-3]), x, iters=3, tau=0.05, sigma=9.8, nu=100.0)
        out.append(x.cpu().numpy().astype(np.float64))
    assert np.linalg.norm(out[1]) > 0
    assert rel(out[0], out[1]) <= 1e-3
