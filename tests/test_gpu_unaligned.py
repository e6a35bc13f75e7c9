"""Device arrays that begin at an odd element (a contiguous view t[1:]): the
entry points promise no more than the alignment of an element."""
import numpy as np
import pytest
import torch

import paper_1502_05037_gb300 as pk
from gpu_util import DEV, rel
from oracle import unet as un
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
