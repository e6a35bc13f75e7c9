"""The half plane and the whole one. A plan with a fixed tile edge is not timed
and runs on the half plane at every size: the operators, the solvers and the
adjoint's lanes of every kernel width there, against the FP64 oracle. Plans of
small images without one take what was faster: right either way, and a second
plan of a shape takes what the first found."""
import numpy as np
import pytest
import torch

import paper_1502_05037_gb300 as pk
from gpu_util import DEV, TOL, np_cplx, np_real, rel, t_cplx, t_real
from oracle import nufft as onf
from oracle import primal_dual as opd
from oracle import sdmm as osd
from paper_1502_05037_gb300 import synth
from test_gpu_half_plane import SHAPES, coverage

pytestmark = pytest.mark.gpu

F32, F64 = pk.PURIFY_F32, pk.PURIFY_F64


def operators(plan, op, nx, ny, M, seed, dtype):
    x = synth.rng(seed).standard_normal((ny, nx)).astype(np_real(dtype))
    xd = torch.from_numpy(x).to(DEV)
    y = torch.empty(M, dtype=t_cplx(dtype), device=DEV)
    a = torch.empty((ny, nx), dtype=t_cplx(dtype), device=DEV)
    n = torch.empty((ny, nx), dtype=t_real(dtype), device=DEV)
    pk.purify_phi(plan, xd, y)
    pk.purify_phi_adj(plan, y, a)
    pk.purify_phi_normal(plan, xd, n)
    want = onf.phi(op, x.astype(np.float64))
    back = onf.phi_adj(op, want)
    # the adjoint of the device's own Phi x: one more rounding of its input
    assert rel(y.cpu(), want) <= TOL[dtype]
    assert rel(a.cpu(), back) <= 2 * TOL[dtype]
    assert rel(n.cpu(), np.real(back)) <= TOL[dtype]


@pytest.mark.parametrize("dtype", [F32, F64])
@pytest.mark.parametrize("J", [2, 3, 4, 5, 6, 7, 8])
@pytest.mark.parametrize("nx,ny,M", [s for s in SHAPES if s[0] < 512])
def test_operators_on_the_half_plane(nx, ny, M, J, dtype):
    u, v = coverage(M, nx + ny + M + J, dtype)
    op = onf.NufftPlan(nx, ny, u.astype(np.float64), v.astype(np.float64), J)
    plan = pk.Plan(nx, ny, torch.from_numpy(u).to(DEV), torch.from_numpy(v).to(DEV), kb_width=J, levels=2,
                   dtype=dtype, tile=16)
    assert plan.info.degrid_mode == 8 and (plan.info.normal_mode in (4, 7) or dtype == F64)
    operators(plan, op, nx, ny, M, J, dtype)


@pytest.mark.parametrize("alpha,n", [(4.0, 16), (4.0, 64), (2.0, 64)])
@pytest.mark.parametrize("dtype", [F32, F64])
def test_half_plane_of_other_oversampling(alpha, n, dtype):
    M, J = 4001, 4
    u, v = coverage(M, n, dtype)
    op = onf.NufftPlan(n, n, u.astype(np.float64), v.astype(np.float64), J, alpha=alpha)
    plan = pk.Plan(n, n, torch.from_numpy(u).to(DEV), torch.from_numpy(v).to(DEV), kb_width=J, levels=2, dtype=dtype,
                   oversample=alpha, tile=16)
    operators(plan, op, n, n, M, n, dtype)


def solves(plan, op, nx, ny, M, J, offs, levels, dtype, tol):
    x_true = np.abs(synth.rng(J).standard_normal((ny, nx)))
    y0 = onf.phi(op, x_true)
    sig = osd.noise_sigma(y0, 30.0)
    y = (y0 + sig * synth.unit_noise(M, J)).astype(np_cplx(dtype)).astype(np.complex128)
    prob = osd.Problem(op, levels, y, offs, osd.epsilon_chi2(sig, np.diff(offs)))
    yd = torch.from_numpy(prob.y.astype(np_cplx(dtype))).to(DEV)
    x = torch.zeros((ny, nx), dtype=t_real(dtype), device=DEV)
    pk.purify_sdmm_solve(plan, yd, prob.eps, x, max_iter=6, cg_iters=5, gamma=prob.gamma, nu=prob.nu)
    assert rel(x.cpu().numpy(), osd.sdmm_solve(prob, np.zeros((ny, nx)), 6, 5).x) <= tol
    x.zero_()
    pk.purify_pd_solve(plan, yd, prob.eps, x, iters=6, tau=0.05, sigma=9.8, nu=prob.nu)
    assert rel(x.cpu().numpy(), opd.chambolle_pock(prob, 6, tau=0.05, sigma=9.8, x0=np.zeros((ny, nx)))) <= tol


@pytest.mark.parametrize("J,dtype,nx,ny", [(8, F32, 32, 16), (7, F32, 16, 32), (6, F32, 64, 32), (2, F64, 16, 16),
                                           (3, F64, 32, 32), (5, F64, 16, 32), (7, F64, 32, 16), (8, F64, 32, 32)])
def test_solves_on_the_half_plane(J, dtype, nx, ny):
    M = 2501
    offs = np.array([0, 700, 701, M])
    u, v = synth.uv_coverage(M, 90 + J, dtype=np_real(dtype))
    op = onf.NufftPlan(nx, ny, u.astype(np.float64), v.astype(np.float64), J)
    plan = pk.Plan(nx, ny, torch.from_numpy(u).to(DEV), torch.from_numpy(v).to(DEV), kb_width=J, levels=2,
                   block_offsets=offs, dtype=dtype, tile=16)
    assert plan.info.degrid_mode == 8
    solves(plan, op, nx, ny, M, J, offs, 2, dtype, 1e-3 if dtype == F32 else 1e-9)


@pytest.mark.parametrize("nx,ny,M,J,dtype", [(64, 64, 2001, 6, F32), (64, 64, 33001, 6, F32), (32, 32, 1500, 4, F32),
                                             (128, 64, 4001, 8, F32), (32, 64, 2001, 5, F64)])
def test_small_plans_take_either_plane(nx, ny, M, J, dtype):
    offs = np.array([0, 700, 701, M])
    u, v = synth.uv_coverage(M, 60 + J, dtype=np_real(dtype))
    op = onf.NufftPlan(nx, ny, u.astype(np.float64), v.astype(np.float64), J)
    ud, vd = torch.from_numpy(u).to(DEV), torch.from_numpy(v).to(DEV)
    modes = []
    for _ in range(2):
        plan = pk.Plan(nx, ny, ud, vd, kb_width=J, levels=2, block_offsets=offs, dtype=dtype)
        modes.append((plan.info.grid_mode, plan.info.degrid_mode, plan.info.normal_mode, plan.info.workspace_bytes))
        operators(plan, op, nx, ny, M, J, dtype)
        solves(plan, op, nx, ny, M, J, offs, 2, dtype, 1e-3 if dtype == F32 else 1e-9)
    assert modes[0] == modes[1]


@pytest.mark.parametrize("dtype", [F32, F64])
def test_a_shape_is_its_grid_too(dtype):
    """Plans of one image and other oversampling do not share launch shapes: a
    block of several short transforms would be one of several thousand threads
    for the long ones."""
    n, M, J = 16, 601, 4
    u, v = coverage(M, 77, dtype)
    ud, vd = torch.from_numpy(u).to(DEV), torch.from_numpy(v).to(DEV)
    for alpha in (2.0, 256.0, 32.0, 2.0):
        op = onf.NufftPlan(n, n, u.astype(np.float64), v.astype(np.float64), J, alpha=alpha)
        plan = pk.Plan(n, n, ud, vd, kb_width=J, levels=2, dtype=dtype, oversample=alpha)
        operators(plan, op, n, n, M, 3, dtype)
