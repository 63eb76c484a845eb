"""The tcgen05 weight and bias gradients at the edges of their 4 x 32 pixel
patches: images lower than a patch, rows left over at one or both levels, a
run of several patches, every block of input channels (16, 32, 64 and several
of 64) and of output channels (32 and 64).  Up to three levels against the FP64
reference of the network, to the bars that hold for whole patches there; at
four, where the bf16 activations' own rounding exceeds those, against the
mma.sync path, to the bars that hold between the two at full size.
"""
import numpy as np
import pytest
import torch

import test_gpu_surrogate as base

pytestmark = pytest.mark.gpu

lib = base.lib


@pytest.mark.parametrize("levels,batch,h,w", [
    (1, 1, 2, 64),     # half a patch high: 16 -> 32 and 32 -> 32 channels
    (1, 2, 5, 128),    # one row left over
    (2, 3, 6, 128),    # two rows left over, and three at the lower level
    (2, 7, 26, 256),   # several patches per run
    (3, 1, 20, 256)])  # 128 channels: two blocks each way
def test_gradients_on_ragged_patches(lib, levels, batch, h, w):
    base.test_forward_and_gradients_match_fp64_reference(lib, levels, batch, h, w, True)


def test_deep_network_follows_the_warp_level_path(lib):
    levels, batch, h, w = 4, 2, 24, 512  # 256 channels, three rows at the lowest level
    rng = np.random.default_rng(levels)
    x = torch.from_numpy(rng.normal(size=(batch, h, w, 4)).astype(np.float32)).cuda()
    t = torch.from_numpy(rng.normal(size=(batch, h, w, 3)).astype(np.float32)).cuda()
    net = lib.UNet(in_ch=4, out_ch=3, base_ch=32, levels=levels, batch=batch, height=h, width=w,
                   seed=7, stream=lib.current_stream())
    g = {}
    for tc in (True, False):
        net.set_tensor_path(tc)
        net.grad(x, t)
        g[tc] = net.grads().astype(np.float64)
    net.close()
    assert base._rel(g[True], g[False]) < 3e-2
    assert base._cos(g[True], g[False]) > 0.9995
