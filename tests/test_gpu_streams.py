"""Plans, solvers and networks made and used on a stream that does not wait for
the default stream: tables uploaded while they are made are there when the
first kernel reads them. The default stream is kept busy meanwhile."""
import numpy as np
import pytest
import torch

import paper_1502_05037_gb300 as pk
from gpu_util import DEV, TOL, np_real, rel, t_real
from oracle import nufft as onf
from oracle import sdmm as osd
from paper_1502_05037_gb300 import synth

pytestmark = pytest.mark.gpu


def busy():
    """A few milliseconds of copies on the default stream."""
    a = torch.empty(1 << 28, dtype=torch.uint8, device=DEV)
    b = torch.empty_like(a)
    for _ in range(20):
        b.copy_(a)
        a.copy_(b)


@pytest.mark.parametrize("n,M,J,dtype,mode", [
    (64, 60001, 6, pk.PURIFY_F32, None), (256, 150001, 6, pk.PURIFY_F32, 7), (64, 60001, 5, pk.PURIFY_F64, 7),
])
def test_plan_and_solver_on_their_own_stream(n, M, J, dtype, mode):
    u, v = synth.uv_coverage(M, 31, dtype=np_real(dtype))
    ud, vd = torch.from_numpy(u).to(DEV), torch.from_numpy(v).to(DEV)
    op = onf.NufftPlan(n, n, u.astype(np.float64), v.astype(np.float64), J)
    x = synth.rng(3).standard_normal((n, n)).astype(np_real(dtype))
    xd, out = torch.from_numpy(x).to(DEV), torch.empty((n, n), dtype=t_real(dtype), device=DEV)
    torch.cuda.synchronize()
    stream = torch.cuda.Stream()
    busy()
    plan = pk.Plan(n, n, ud, vd, kb_width=J, levels=2, dtype=dtype, stream=stream)
    assert mode is None or plan.info.normal_mode == mode
    pk.purify_phi_normal(plan, xd, out)
    stream.synchronize()
    y = onf.phi(op, x.astype(np.float64))
    assert rel(out.cpu(), np.real(onf.phi_adj(op, y))) <= TOL[dtype]


@pytest.mark.parametrize("groups", [0, 2])
def test_solve_on_its_own_stream(groups):
    n, M, J, levels, tol = 32, 3000, 4, 2, 1e-3
    u, v = synth.uv_coverage(M, 32, dtype=np.float32)
    offs = np.array([0, 700, 1500, 2200, M])
    op = onf.NufftPlan(n, n, u.astype(np.float64), v.astype(np.float64), J)
    y0 = onf.phi(op, np.abs(synth.rng(4).standard_normal((n, n))))
    sig = osd.noise_sigma(y0, 30.0)
    y = (y0 + sig * synth.unit_noise(M, 5)).astype(np.complex64)
    prob = osd.Problem(op, levels, y.astype(np.complex128), offs, osd.epsilon_chi2(sig, np.diff(offs)))
    ud, vd = torch.from_numpy(u).to(DEV), torch.from_numpy(v).to(DEV)
    yd = torch.from_numpy(prob.y.astype(np.complex64)).to(DEV)
    got = []
    for own in (False, True):
        x = torch.zeros((n, n), dtype=torch.float32, device=DEV)
        torch.cuda.synchronize()
        stream = torch.cuda.Stream() if own else None
        plan = pk.Plan(n, n, ud, vd, kb_width=J, levels=levels, block_offsets=offs, stream=stream)
        busy()
        seq = [i % 2 for i in range(6)] if groups else None
        pk.purify_sdmm_solve(plan, yd, prob.eps, x, max_iter=6, cg_iters=5, gamma=prob.gamma, nu=prob.nu,
                             block_groups=groups, group_seq=seq)
        torch.cuda.synchronize()
        got.append(x.cpu().numpy())
    if not groups:
        assert rel(got[1], osd.sdmm_solve(prob, np.zeros((n, n)), 6, 5).x) <= tol
    assert rel(got[1], got[0]) <= tol


def test_network_on_its_own_stream():
    x = torch.randn((1, 32, 32), dtype=torch.float32, device=DEV)
    outs = []
    for own in (False, True):
        torch.cuda.synchronize()
        stream = torch.cuda.Stream() if own else None
        busy()
        net = pk.Unet(32, 32, 2, 16, max_batch=1, seed=4, stream=stream)
        y = torch.empty_like(x)
        torch.cuda.synchronize()
        net.forward(x, y)
        torch.cuda.synchronize()
        outs.append(y.cpu())
    assert torch.equal(outs[0], outs[1])
