"""The tiled convolution and weight-gradient kernels at the edges of their
tiles: images that are no multiple of 16 x 8, channel counts between the
16-channel steps, inputs too wide for a staged tile, and a network whose
levels end inside a tile. Tolerances as in test_gpu_unet.py (same rounding
points, FP32 accumulation)."""
import numpy as np
import pytest
import torch

import paper_1502_05037_gb300 as pk
from gpu_util import DEV, rel
from oracle import unet as un
from test_gpu_unet import bf16_round, flat_from_oracle, oracle_params_from_flat

pytestmark = pytest.mark.gpu


@pytest.mark.parametrize("B,H,W,Cin,Cout,k", [
    (1, 1, 1, 8, 16, 3),
    (3, 17, 9, 24, 40, 3),       # one row and one column past a tile
    (1, 15, 7, 3, 5, 3),         # channels copied one by one
    (2, 33, 24, 40, 24, 1),
    (1, 16, 8, 416, 256, 3),     # the widest staged input
    (1, 10, 12, 432, 32, 3),     # gathered tap by tap
    (1, 40, 40, 128, 256, 3),    # output channels split over blocks
])
def test_conv_tiles(B, H, W, Cin, Cout, k):
    g = np.random.default_rng(H * 100 + W + Cin)
    x = g.standard_normal((B, H, W, Cin)).astype(np.float32)
    w = (g.standard_normal((Cout, k, k, Cin)) / np.sqrt(k * k * Cin)).astype(np.float32)
    b = g.standard_normal(Cout).astype(np.float32)
    out = torch.empty((B, H, W, Cout), dtype=torch.float32, device=DEV)
    pk.purify_conv2d(torch.from_numpy(x).to(DEV), torch.from_numpy(w).to(DEV), torch.from_numpy(b).to(DEV), out, k)
    assert rel(out.cpu().numpy(), un.conv2d(bf16_round(x), bf16_round(w), b.astype(np.float64))) <= 1e-5


@pytest.mark.parametrize("H,W,levels,base,B", [(24, 40, 3, 24, 2), (12, 20, 2, 40, 1)])
def test_gradients_on_partial_tiles(H, W, levels, base, B):
    net = pk.Unet(H, W, levels, base, max_batch=B, seed=H + W)
    flat = np.empty(net.num_params, dtype=np.float32)
    net.get_params(flat)
    params = oracle_params_from_flat(flat, levels, base)
    g = np.random.default_rng(7)
    x = g.standard_normal((B, H, W)).astype(np.float32)
    t = g.standard_normal((B, H, W)).astype(np.float32)
    grads = torch.empty(net.num_params, dtype=torch.float32, device=DEV)
    xd, td = torch.from_numpy(x).to(DEV), torch.from_numpy(t).to(DEV)
    loss = net.gradients(xd, td, grads)
    pred, cache = un.forward(params, x[..., None].astype(np.float64), levels, base, q=bf16_round)
    want_loss, gpred = un.mse(pred, t[..., None].astype(np.float64))
    assert abs(loss - want_loss) <= 1e-3 * want_loss
    want = un.backward(params, x[..., None].astype(np.float64), cache, gpred, levels, base)
    got = oracle_params_from_flat(grads.cpu().numpy(), levels, base)
    errs = {k: rel(got[k], want[k]) for k in want if np.linalg.norm(want[k]) > 0}
    bad = {k: round(e, 4) for k, e in errs.items() if e > 3e-2}
    assert not bad, bad
    assert rel(flat_from_oracle(got, levels, base), flat_from_oracle(want, levels, base)) <= 1.5e-2


@pytest.mark.parametrize("B,H,W,Cin,Cout,k", [
    (41, 70, 45, 32, 64, 3),     # several tiles a block, a last round that is not full
    (60, 33, 41, 16, 16, 1),
    (12, 70, 90, 8, 128, 3),
])
def test_blocks_that_walk_tiles(B, H, W, Cin, Cout, k):
    """A block's second and later tiles are the same sums in the same order as
    one image alone, where every block has one tile: equal to the bit."""
    g = np.random.default_rng(B)
    x = torch.from_numpy(g.standard_normal((B, H, W, Cin)).astype(np.float32)).to(DEV)
    w = torch.from_numpy((g.standard_normal((Cout, k, k, Cin)) / np.sqrt(k * k * Cin)).astype(np.float32)).to(DEV)
    b = torch.from_numpy(g.standard_normal(Cout).astype(np.float32)).to(DEV)
    out = torch.empty((B, H, W, Cout), dtype=torch.float32, device=DEV)
    one = torch.empty((1, H, W, Cout), dtype=torch.float32, device=DEV)
    pk.purify_conv2d(x, w, b, out, k)
    for i in (0, 1, B // 2, B - 1):
        pk.purify_conv2d(x[i:i + 1].contiguous(), w, b, one, k)
        assert torch.equal(out[i], one[0]), i
