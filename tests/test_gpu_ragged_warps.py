"""Convolutions and weight gradients where a warp's lanes differ at every step of
an epilogue: rows of a tile outside the image beside rows inside it, output
channels that end inside a warp's 32 rows of an accumulator. Tolerances as in
test_gpu_unet.py."""
import numpy as np
import pytest
import torch

import paper_1502_05037_gb300 as pk
from gpu_util import DEV, rel
from oracle import unet as un
from test_gpu_unet import bf16_round, oracle_params_from_flat

pytestmark = pytest.mark.gpu


@pytest.mark.parametrize("W", [1, 3, 5, 7])
@pytest.mark.parametrize("Cin,Cout", [(16, 1), (24, 17), (8, 72), (432, 40)])
def test_conv_rows_outside_the_image(W, Cin, Cout):
    B, H, k = 2, 5, 3
    g = np.random.default_rng(W + Cin)
    x = g.standard_normal((B, H, W, Cin)).astype(np.float32)
    w = (g.standard_normal((Cout, k, k, Cin)) / np.sqrt(k * k * Cin)).astype(np.float32)
    b = g.standard_normal(Cout).astype(np.float32)
    out = torch.empty((B, H, W, Cout), dtype=torch.float32, device=DEV)
    pk.purify_conv2d(torch.from_numpy(x).to(DEV), torch.from_numpy(w).to(DEV), torch.from_numpy(b).to(DEV), out, k)
    assert rel(out.cpu().numpy(), un.conv2d(bf16_round(x), bf16_round(w), b.astype(np.float64))) <= 1e-5


@pytest.mark.parametrize("base", [8, 24, 40])
def test_weight_gradients_of_channels_within_a_warp(base):
    H, W, levels, B = 20, 12, 2, 3
    net = pk.Unet(H, W, levels, base, max_batch=B, seed=base)
    flat = np.empty(net.num_params, dtype=np.float32)
    net.get_params(flat)
    params = oracle_params_from_flat(flat, levels, base)
    g = np.random.default_rng(base)
    x = g.standard_normal((B, H, W)).astype(np.float32)
    t = g.standard_normal((B, H, W)).astype(np.float32)
    grads = torch.empty(net.num_params, dtype=torch.float32, device=DEV)
    net.gradients(torch.from_numpy(x).to(DEV), torch.from_numpy(t).to(DEV), grads)
    pred, cache = un.forward(params, x[..., None].astype(np.float64), levels, base, q=bf16_round)
    _, gpred = un.mse(pred, t[..., None].astype(np.float64))
    want = un.backward(params, x[..., None].astype(np.float64), cache, gpred, levels, base)
    got = oracle_params_from_flat(grads.cpu().numpy(), levels, base)
    bad = {n: round(rel(got[n], want[n]), 4) for n in want if np.linalg.norm(want[n]) > 0 and rel(got[n], want[n]) > 3e-2}
    assert not bad, bad
