"""The half-plane path of autotuned plans (Phi, the normal operator as a
stencil or over lane pairs, the solver's adjoint through the normal operator)
against the FP64 oracle: the smallest grids, rectangular and wrapped
footprints, every kernel width, one visibility, dense cells and an image too
sparse for the stencil."""
import numpy as np
import pytest
import torch

import paper_1502_05037_gb300 as pk
from gpu_util import DEV, TOL, np_cplx, np_real, rel, t_cplx, t_real
from oracle import nufft as onf
from paper_1502_05037_gb300 import synth

pytestmark = pytest.mark.gpu

SHAPES = [
    (8, 8, 1), (8, 16, 40), (16, 8, 2001),      # the half plane is wider than the grid
    (32, 64, 3001), (64, 16, 517),              # rectangular, columns past the last block
    (64, 64, 60001),                            # many visibilities per cell
    (512, 512, 3001),                           # sparse: lane pairs in FP32
]


def coverage(M, seed, dtype):
    """Uniform coverage with the corners of [-pi, pi) and zero among it
    (footprints across both halves and the periodic edges). Other points on
    grid lines are left out: there the FP32 split and FP64 may pick footprints
    one cell apart."""
    u, v = synth.uv_coverage(M, seed, uniform_fraction=1.0, dtype=np_real(dtype))
    top = np.nextafter(np_real(dtype)(np.pi), np_real(dtype)(0))
    edge = np.array([1e-3, 0.0, -top, top, -1e-3, -0.0], dtype=u.dtype)
    n = min(M, edge.size)
    u[:n], v[:n] = edge[:n], edge[::-1][:n]
    if M >= 2 * edge.size:
        u[n:2 * n], v[n:2 * n] = edge, edge
    return u, v


@pytest.mark.parametrize("dtype", [pk.PURIFY_F32, pk.PURIFY_F64])
@pytest.mark.parametrize("J", [2, 3, 4, 5, 6, 7, 8])
@pytest.mark.parametrize("nx,ny,M", SHAPES)
def test_half_plane_operators(nx, ny, M, J, dtype):
    if nx == 512 and (dtype == pk.PURIFY_F64 or J not in (5, 6, 8)):
        pytest.skip("one sparse size is enough")
    u, v = coverage(M, nx + ny + M + J, dtype)
    op = onf.NufftPlan(nx, ny, u.astype(np.float64), v.astype(np.float64), J)
    plan = pk.Plan(nx, ny, torch.from_numpy(u).to(DEV), torch.from_numpy(v).to(DEV), kb_width=J, levels=2,
                   dtype=dtype)
    if nx == 512:
        assert plan.info.normal_mode == 4
    x = synth.rng(J).standard_normal((ny, nx)).astype(np_real(dtype))
    xd = torch.from_numpy(x).to(DEV)
    y = torch.empty(M, dtype=t_cplx(dtype), device=DEV)
    n = torch.empty((ny, nx), dtype=t_real(dtype), device=DEV)
    pk.purify_phi(plan, xd, y)
    pk.purify_phi_normal(plan, xd, n)
    want = onf.phi(op, x.astype(np.float64))
    assert rel(y.cpu(), want) <= TOL[dtype]
    assert rel(n.cpu(), np.real(onf.phi_adj(op, want))) <= TOL[dtype]
    # a second pass finds clean accumulators
    pk.purify_phi_normal(plan, xd, n)
    assert rel(n.cpu(), np.real(onf.phi_adj(op, want))) <= TOL[dtype]


@pytest.mark.parametrize("dtype", [pk.PURIFY_F32, pk.PURIFY_F64])
def test_half_plane_keeps_every_visibility_in_place(dtype):
    # unit images: each visibility's own phase, conjugated where it was folded
    n, M, J = 16, 777, 6
    u, v = coverage(M, 5, dtype)
    plan = pk.Plan(n, n, torch.from_numpy(u).to(DEV), torch.from_numpy(v).to(DEV), kb_width=J, levels=2,
                   block_offsets=np.array([0, 1, 300, M]), dtype=dtype)
    op = onf.NufftPlan(n, n, u.astype(np.float64), v.astype(np.float64), J)
    for i, j in ((0, 0), (3, 15), (8, 8)):
        x = np.zeros((n, n), dtype=np_real(dtype))
        x[i, j] = 1.0
        y = torch.empty(M, dtype=t_cplx(dtype), device=DEV)
        pk.purify_phi(plan, torch.from_numpy(x).to(DEV), y)
        got, want = y.cpu().numpy(), onf.phi(op, x.astype(np.float64))
        assert np.abs(got - want.astype(np_cplx(dtype))).max() <= 10 * TOL[dtype] * np.abs(want).max()
