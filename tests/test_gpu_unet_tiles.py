"""The tile geometries and ring depths of the 3x3x3 convolution and of its
weight gradient against FP64.

Inputs are BF16-representable, so every product is exact and only FP32 sums
round: of at most 27 x 64 terms for an output (relative L2 error <= 1e-5), and
for a weight of up to 25600 products, added 16 at a time in runs of at most
two tiles and then by atomics (sqrt(25600) 2^-24 = 1e-5; <= 2e-5).  The same for
the bias gradient."""
import ctypes as C

import numpy as np
import pytest

pytestmark = pytest.mark.gpu

SHAPES = [(1, 2, 8, 64),      # rows of 64: tiles of 4 rows of 32
          (1, 2, 4, 256),
          (1, 2, 6, 64),      # a height that tiles of 4 rows do not divide: boxes of single voxels
          (2, 50, 16, 16),    # more tiles than SMs: the short ring
          (5, 2, 4, 4),       # whole samples per tile, a partial last tile
          (3, 8, 4, 8),       # parts of one sample per tile
          (3, 3, 4, 4)]       # tiles that cut samples: plane by plane


def _ptr(t):
    return C.c_void_p(t.data_ptr())


def _shifts(x):
    """x moved by every tap, zeros outside the sample: (27, n, D, H, W, c)."""
    import torch
    p = torch.nn.functional.pad(x, (0, 0, 1, 1, 1, 1, 1, 1))
    n, D, H, W, _ = x.shape
    return [p[:, t // 9:t // 9 + D, t // 3 % 3:t // 3 % 3 + H, t % 3:t % 3 + W] for t in range(27)]


@pytest.mark.parametrize("cin,cout", [(16, 16), (64, 32)])
@pytest.mark.parametrize("shape", SHAPES)
def test_tiles_and_rings(shape, cin, cout):
    import torch
    import paper_1711_04471_gb300 as P
    P.build()
    from paper_1711_04471_gb300 import _native as N
    g = torch.Generator(device="cuda").manual_seed(7)

    def rnd(*s):
        return torch.randn(s, device="cuda", generator=g).to(torch.bfloat16).float()

    n, D, H, W = shape
    x, w, gy = rnd(*shape, cin), rnd(27, cout, cin) * 0.25, rnd(*shape, cout)
    y, b = torch.empty_like(gy), torch.zeros(cout, device="cuda")
    dw, db = torch.empty_like(w), torch.empty(cout, device="cuda")
    torch.cuda.synchronize()
    N.check(N.lib().unet_conv3d(n, D, H, W, cin, cout, _ptr(x), _ptr(w), _ptr(b), 1, None, _ptr(y), None), "conv")
    N.check(N.lib().unet_conv3d_bwd_weight(n, D, H, W, cin, cout, _ptr(x), _ptr(gy), _ptr(dw), _ptr(db), None), "wgrad")
    torch.cuda.synchronize()
    xs = [s.double() for s in _shifts(x)]
    ry = sum(s @ w[t].double().T for t, s in enumerate(xs))
    rw = torch.stack([torch.einsum("nzyxo,nzyxi->oi", gy.double(), s) for s in xs])
    rel = lambda a, r: float((a.double() - r).norm() / r.norm())
    assert rel(y, ry) <= 1e-5
    assert rel(dw, rw) <= 2e-5
    assert np.allclose(db.cpu().numpy(), gy.double().sum((0, 1, 2, 3)).cpu().numpy(), rtol=0, atol=2e-5 * (n * D * H * W) ** 0.5)
