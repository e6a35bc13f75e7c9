"""The solver's data-side kernels at their edges against the FP64 oracle: blocks
of one and a few visibilities and blocks that begin and end at odd places
(chunks are read two visibilities at a time), and the adjoint over runs of
every kernel width on rectangular grids. Tolerances as in test_gpu_sdmm.py."""
import numpy as np
import pytest
import torch

import paper_1502_05037_gb300 as pk
from gpu_util import DEV, np_cplx, np_real, rel, t_real
from oracle import nufft as onf
from oracle import primal_dual as opd
from oracle import sdmm as osd
from paper_1502_05037_gb300 import synth

pytestmark = pytest.mark.gpu

SIZES = [1, 1, 2, 3, 4095, 1, 4097, 700]


@pytest.mark.parametrize("nx,ny,J,dtype", [
    (32, 32, 2, pk.PURIFY_F32), (32, 16, 3, pk.PURIFY_F32), (16, 32, 4, pk.PURIFY_F32), (32, 64, 5, pk.PURIFY_F32),
    (64, 32, 6, pk.PURIFY_F32), (32, 32, 7, pk.PURIFY_F32), (32, 16, 6, pk.PURIFY_F64),
])
def test_uneven_blocks(nx, ny, J, dtype):
    M, levels, tol = sum(SIZES), 2, 1e-3 if dtype == pk.PURIFY_F32 else 1e-9
    offs = np.concatenate([[0], np.cumsum(SIZES)])
    u, v = synth.uv_coverage(M, 70 + J, dtype=np_real(dtype))
    plan = pk.Plan(nx, ny, torch.from_numpy(u).to(DEV), torch.from_numpy(v).to(DEV), kb_width=J, levels=levels,
                   block_offsets=offs, dtype=dtype)
    op = onf.NufftPlan(nx, ny, u.astype(np.float64), v.astype(np.float64), J)
    x_true = np.abs(synth.rng(J).standard_normal((ny, nx)))
    y0 = onf.phi(op, x_true)
    sig = osd.noise_sigma(y0, 30.0)
    y = (y0 + sig * synth.unit_noise(M, J)).astype(np_cplx(dtype)).astype(np.complex128)
    prob = osd.Problem(op, levels, y, offs, osd.epsilon_chi2(sig, np.diff(offs)))
    yd = torch.from_numpy(prob.y.astype(np_cplx(dtype))).to(DEV)
    x = torch.zeros((ny, nx), dtype=t_real(dtype), device=DEV)
    ref = osd.sdmm_solve(prob, np.zeros((ny, nx)), 8, 6).x
    st = pk.purify_sdmm_solve(plan, yd, prob.eps, x, max_iter=8, cg_iters=6, gamma=prob.gamma, nu=prob.nu)
    assert rel(x.cpu().numpy(), ref) <= tol
    assert abs(st.max_resid_over_eps - osd.residual_ratios(prob, ref).max()) <= 10 * tol * max(
        1.0, osd.residual_ratios(prob, ref).max())
    x.zero_()
    ref = opd.chambolle_pock(prob, 8, tau=0.05, sigma=9.8, x0=np.zeros((ny, nx)))
    pk.purify_pd_solve(plan, yd, prob.eps, x, iters=8, tau=0.05, sigma=9.8, nu=prob.nu)
    assert rel(x.cpu().numpy(), ref) <= tol
