"""Tiles of several planes (small planes) at depths that neither divide the
tile's planes nor are divided by them: the last tile of a sample holds planes
past its end, which are zero fill and not stored.  Against FP64 with the
bounds of test_gpu_unet_tiles, and a batch against its samples one by one: a
voxel's sums run over the same products in the same order, so they are equal."""
import numpy as np
import pytest

import test_gpu_unet_tiles as tiles

pytestmark = pytest.mark.gpu


@pytest.mark.parametrize("cin,cout", [(16, 16), (64, 32)])
@pytest.mark.parametrize("shape", [(2, 12, 4, 4),    # 8 planes a tile: one and a half tiles a sample
                                   (1, 1, 4, 8),     # one plane of four
                                   (40, 3, 4, 4),    # three planes of eight, many samples
                                   (3, 5, 8, 8),     # 2 planes a tile
                                   (2, 9, 4, 16),
                                   (2, 6, 2, 8),
                                   (3, 31, 4, 8)])
def test_depths_that_do_not_divide(shape, cin, cout):
    tiles.test_tiles_and_rings(shape, cin, cout)


@pytest.mark.parametrize("D,H", [(12, 16), (20, 16), (60, 16), (12, 32), (28, 32)])
def test_forward_of_a_batch_is_that_of_its_samples(D, H):
    import torch
    import paper_1711_04471_gb300 as P
    P.build()
    from paper_1711_04471_gb300.unet import UNet
    x = torch.randn((3, D, H, H, 2), device="cuda", generator=torch.Generator(device="cuda").manual_seed(D))
    with UNet(seed=1) as net:
        whole = net.forward(x).cpu().numpy()
        for k in range(3):
            assert np.array_equal(net.forward(x[k:k + 1].contiguous()).cpu().numpy()[0], whole[k])
