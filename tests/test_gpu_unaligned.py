"""Device arrays that begin at an odd element (a contiguous view t[1:]): the
entry points promise no more than the alignment of an element."""
import numpy as np
import pytest
import torch

import paper_1502_05037_gb300 as pk
from gpu_util import DEV, TOL, make_plan, np_real, rel, t_real
from oracle import unet as un
from oracle import wavelets as ow
from paper_1502_05037_gb300 import synth
from test_gpu_unet import bf16_round

pytestmark = pytest.mark.gpu


def shifted(shape, dtype, first=1):
    """An uninitialised contiguous device array whose first element is element
    `first` of its allocation."""
    n = int(np.prod(shape))
    return torch.empty(n + first, dtype=dtype, device=DEV)[first:].view(shape)


@pytest.mark.parametrize("first", [1, 2, 3])
@pytest.mark.parametrize("Cin,Cout", [(16, 16), (24, 64), (432, 32)])
def test_conv2d_output_at_an_odd_element(Cin, Cout, first):
    B, H, W, k = 1, 9, 17, 3
    g = np.random.default_rng(Cin)
    x = g.standard_normal((B, H, W, Cin)).astype(np.float32)
    w = (g.standard_normal((Cout, k, k, Cin)) / np.sqrt(k * k * Cin)).astype(np.float32)
    b = g.standard_normal(Cout).astype(np.float32)
    args = []
    for a in (x, w, b):
        t = shifted(a.shape, torch.float32, first)
        t.copy_(torch.from_numpy(a))
        args.append(t)
    out = shifted((B, H, W, Cout), torch.float32, first)
    assert out.data_ptr() % 16 == 4 * first and out.is_contiguous()
    pk.purify_conv2d(*args, out, k)
    assert rel(out.cpu().numpy(), un.conv2d(bf16_round(x), bf16_round(w), b.astype(np.float64))) <= 1e-5


@pytest.mark.parametrize("dtype", [pk.PURIFY_F32, pk.PURIFY_F64])
@pytest.mark.parametrize("nx,ny,levels,mask", [
    (128, 64, 3, 0x1FF), (64, 256, 2, 0x1FE), (16, 512, 3, 0x1FF), (256, 256, 4, 0x107),
])
def test_dictionary_of_arrays_at_an_odd_element(nx, ny, levels, mask, dtype):
    plan, *_ = make_plan(nx, ny, 64, 4, levels=levels, dtype=dtype, mask=mask)
    rt, q, tol = t_real(dtype), bin(mask).count("1"), TOL[dtype]
    g = synth.rng(nx + levels)
    x = g.standard_normal((ny, nx)).astype(np_real(dtype))
    c = g.standard_normal((q, ny, nx)).astype(np_real(dtype))
    want_c = ow.psi_adj(x.astype(np.float64), levels, mask)
    want_x = ow.psi(c.astype(np.float64), levels, mask)
    for first in (1, 2, 3) if dtype == pk.PURIFY_F32 else (1,):
        xs, cs = shifted(x.shape, rt, first), shifted(c.shape, rt, first)
        xs.copy_(torch.from_numpy(x))
        cs.copy_(torch.from_numpy(c))
        assert xs.data_ptr() % 16 and cs.data_ptr() % 16
        got_c, got_x = shifted(c.shape, rt, first), shifted(x.shape, rt, first)
        pk.purify_psi_adj(plan, xs, got_c)
        assert rel(got_c.cpu(), want_c) <= tol
        pk.purify_psi(plan, cs, got_x)
        assert rel(got_x.cpu(), want_x) <= tol
        pk.purify_reweight(plan, xs, 0.1, got_c)
        assert rel(got_c.cpu(), 0.1 / (0.1 + np.abs(want_c))) <= tol
        assert abs(pk.purify_coef_std(plan, xs) - want_c.std()) <= tol * want_c.std()
        got_c.zero_()
        torch.cuda.synchronize()
        pk.purify_psi_adj_static(xs, got_c, nx, ny, levels, mask, dtype)
        torch.cuda.synchronize()
        assert rel(got_c.cpu(), want_c) <= tol


@pytest.mark.parametrize("nx,ny", [(512, 256), (256, 16)])
def test_transform_of_a_grid_at_an_odd_element(nx, ny):
    plan, *_ = make_plan(nx, ny, 64, 4, levels=2)
    Kx, Ky = plan.info.Kx, plan.info.Ky
    g = synth.rng(nx)
    x = (g.standard_normal((Ky, Kx)) + 1j * g.standard_normal((Ky, Kx))).astype(np.complex64)
    grid = shifted((Ky, Kx), torch.complex64)
    assert grid.data_ptr() % 16 == 8
    for inverse in (False, True):
        grid.copy_(torch.from_numpy(x))
        pk.purify_fft2(plan, grid, inverse)
        ref = np.fft.ifft2(x.astype(np.complex128)) * Kx * Ky if inverse else np.fft.fft2(x.astype(np.complex128))
        assert rel(grid.cpu(), ref) <= TOL[pk.PURIFY_F32]
