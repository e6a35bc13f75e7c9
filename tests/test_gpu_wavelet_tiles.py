"""Analysis and synthesis at the edges of their tiles and tails: bands narrower
than a tile or a filter, rectangular images whose coarse bands end up a few
samples wide, tails that hold all levels or only some, one basis, the Dirac
plane alone, one level - against the FP64 oracle."""
import numpy as np
import pytest
import torch

import paper_1502_05037_gb300 as pk
from gpu_util import DEV, TOL, make_plan, np_real, rel, t_real
from oracle import wavelets as ow
from paper_1502_05037_gb300 import synth

pytestmark = pytest.mark.gpu


@pytest.mark.parametrize("dtype", [pk.PURIFY_F32, pk.PURIFY_F64])
@pytest.mark.parametrize("nx,ny,levels,mask", [
    (8, 8, 1, 0x1FF), (8, 8, 3, 0x1FF), (8, 512, 3, 0x1FF), (512, 8, 3, 0x1FF), (64, 32, 5, 0x1FF),
    (128, 128, 1, 0x1FF), (128, 128, 4, 0x102), (256, 128, 2, 0x100), (256, 256, 7, 0x1FE), (512, 256, 4, 0x01F),
    (64, 64, 2, 0x001), (1024, 16, 4, 0x155),
])
def test_transforms(nx, ny, levels, mask, dtype):
    plan, *_ = make_plan(nx, ny, 64, 4, levels=levels, dtype=dtype, mask=mask)
    g = synth.rng(nx + ny + levels)
    x = g.standard_normal((ny, nx)).astype(np_real(dtype))
    q = bin(mask).count("1")
    c = g.standard_normal((q, ny, nx)).astype(np_real(dtype))
    got_c = torch.empty((q, ny, nx), dtype=t_real(dtype), device=DEV)
    got_x = torch.empty((ny, nx), dtype=t_real(dtype), device=DEV)
    pk.purify_psi_adj(plan, torch.from_numpy(x).to(DEV), got_c)
    pk.purify_psi(plan, torch.from_numpy(c).to(DEV), got_x)
    assert rel(got_c.cpu(), ow.psi_adj(x.astype(np.float64), levels, mask)) <= TOL[dtype]
    assert rel(got_x.cpu(), ow.psi(c.astype(np.float64), levels, mask)) <= TOL[dtype]
    if nx * ny <= 256 * 256:
        torch.cuda.synchronize()
        pk.purify_psi_adj_static(torch.from_numpy(x).to(DEV), got_c, nx, ny, levels, mask, dtype)
        torch.cuda.synchronize()
        assert rel(got_c.cpu(), ow.psi_adj(x.astype(np.float64), levels, mask)) <= TOL[dtype]


@pytest.mark.parametrize("dtype", [pk.PURIFY_F32, pk.PURIFY_F64])
@pytest.mark.parametrize("nx,ny,levels,mask", [
    # either side of each choice of the finest synthesis: by 16-row tiles of 32 columns (FP32) or 8 (FP64)
    (512, 256, 2, 0x1FF), (512, 512, 2, 0x1FF), (1024, 512, 2, 0x1FF),
    (128, 128, 2, 0x1FF), (512, 64, 2, 0x1FF), (256, 256, 2, 0x1FF), (32, 2048, 2, 0x0FF),
    # fewer bases than groups, and filters shorter than the longest beside it
    (64, 64, 2, 0x100), (64, 64, 2, 0x181), (512, 512, 1, 0x00E), (1024, 512, 1, 0x102),
    # one level below the finest in a band that fits the tail, several levels there
    (32, 32, 2, 0x1FF), (16, 16, 3, 0x1FE), (16, 64, 2, 0x1FF), (8, 1024, 2, 0x1FF),
])
def test_synthesis_and_analysis_by_every_tile(nx, ny, levels, mask, dtype):
    plan, *_ = make_plan(nx, ny, 64, 4, levels=levels, dtype=dtype, mask=mask)
    g = synth.rng(3 * nx + ny + levels)
    x = g.standard_normal((ny, nx)).astype(np_real(dtype))
    c = g.standard_normal((bin(mask).count("1"), ny, nx)).astype(np_real(dtype))
    got_c = torch.empty(c.shape, dtype=t_real(dtype), device=DEV)
    got_x = torch.empty((ny, nx), dtype=t_real(dtype), device=DEV)
    pk.purify_psi_adj(plan, torch.from_numpy(x).to(DEV), got_c)
    pk.purify_psi(plan, torch.from_numpy(c).to(DEV), got_x)
    assert rel(got_c.cpu(), ow.psi_adj(x.astype(np.float64), levels, mask)) <= TOL[dtype]
    assert rel(got_x.cpu(), ow.psi(c.astype(np.float64), levels, mask)) <= TOL[dtype]
