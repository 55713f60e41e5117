"""Weight gradient of the 3x3x3 convolution around the edges of its 8 x 16 x 2 voxel tiles and
of the split of the tiles over blocks, against float64, and the bounded wait."""
import numpy as np
import pytest
import torch

import paper_2604_06257_gb300 as m
from paper_2604_06257_gb300 import nn

pytestmark = pytest.mark.gpu


def reference(x, g):
    """(dW, sum |x| |g|) in float64, taps (z, y, x)."""
    d, h, w = x.shape[1:4]
    out = []
    for a, b in ((x.double(), g.double()), (x.double().abs(), g.double().abs())):
        xp = torch.nn.functional.pad(a, (0, 0, 1, 1, 1, 1, 1, 1))
        bb = b.reshape(-1, g.shape[-1])
        out.append(torch.stack([xp[:, i:i + d, j:j + h, k:k + w].reshape(-1, x.shape[-1]).T @ bb
                                for i in range(3) for j in range(3) for k in range(3)]))
    return out


@pytest.mark.parametrize("shape", [(1, 1, 1, 1), (2, 2, 16, 8), (1, 3, 17, 9), (3, 5, 33, 25), (2, 4, 15, 7),
                                   (2, 40, 64, 48)])
@pytest.mark.parametrize("ci,co", [(16, 16), (48, 16), (32, 64)])
def test_weight_gradient_tile_edges(shape, ci, co):
    gen = torch.Generator(device="cuda").manual_seed(sum(shape) + ci + co)
    x = torch.randn(shape + (ci,), device="cuda", generator=gen).to(torch.bfloat16)
    g = torch.randn(shape + (co,), device="cuda", generator=gen).to(torch.bfloat16)
    dw = torch.full((27, ci, co), 0.5, device="cuda")           # the call adds to what is there
    nn.mach_nn_conv3d_wgrad(x, g, dw)
    torch.cuda.synchronize()
    ref, mag = reference(x, g)
    # one rounding of 2^-24 a term at most, and the added 0.5; a chain of roundings is a quarter of a
    # block's voxels and then the blocks' atomics, for the large shape far below 65536
    M = int(np.prod(shape))
    bound = (min(M, 65536) + 64) * 2.0 ** -24 * mag + 2.0 ** -24
    assert bool(((dw.double() - 0.5 - ref).abs() <= bound).all())


def test_weight_gradient_bounded_wait_reports_timeout():
    """Copies announced to nobody: every wait runs out, the kernel sets the error word and
    returns, and the next call is right."""
    x = torch.ones((1, 4, 16, 16, 16), device="cuda", dtype=torch.bfloat16)
    dw = torch.zeros((27, 16, 16), device="cuda")
    lib = m.lib()
    lib.mach_nn_debug_conv(1, 2000)
    try:
        nn.mach_nn_conv3d_wgrad(x, x, dw)
        assert lib.mach_nn_device_status(None) == m.MACH_ERR_TIMEOUT
    finally:
        lib.mach_nn_debug_conv(0, 0)
    dw.zero_()
    nn.mach_nn_conv3d_wgrad(x, x, dw)
    torch.cuda.synchronize()
    assert lib.mach_nn_device_status(None) == m.MACH_OK
    ref, _ = reference(x, x)
    assert torch.equal(dw.double(), ref)
