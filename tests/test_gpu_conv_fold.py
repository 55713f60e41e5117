"""Convolutions of 32 output channels (data gradients x-folded) around the edges of their 14 x 8 voxel
tiles, forward and as data gradient with the leaky ReLU's derivative left to the caller,
against float64 and the 27-tap kernel."""
import pytest
import torch

from paper_2604_06257_gb300 import nn

pytestmark = pytest.mark.gpu


def conv64(x, w):
    k = w.view(3, 3, 3, *w.shape[1:]).permute(4, 3, 0, 1, 2)
    return torch.nn.functional.conv3d(x.permute(0, 4, 1, 2, 3), k, padding=1).permute(0, 2, 3, 4, 1)


@pytest.mark.parametrize("shape", [(1, 1, 1, 1), (2, 3, 8, 14), (1, 2, 9, 15), (2, 5, 7, 29), (3, 4, 33, 13)])
@pytest.mark.parametrize("ci,co", [(16, 32), (32, 32), (48, 32), (96, 32)])
@pytest.mark.parametrize("flip", [False, True])
def test_folded_wide_convolution(shape, ci, co, flip):
    gen = torch.Generator(device="cuda").manual_seed(sum(shape) * ci + co)
    x = torch.randn(shape + (ci,), device="cuda", generator=gen).to(torch.bfloat16)
    # flip: the data gradient of a co -> ci convolution, a convolution with mirrored taps
    w = (torch.randn((27, co, ci) if flip else (27, ci, co), device="cuda", generator=gen) * 0.1).to(torch.bfloat16).float()
    b = torch.randn(co, device="cuda", generator=gen)
    if flip:
        _, pk = nn.mach_nn_pack_weights(w, co, ci, forward=False)
        wk = w.flip(0).transpose(1, 2)
    else:
        pk, _ = nn.mach_nn_pack_weights(w, ci, co, flipped=False)
        wk = w
    ref, mag = conv64(x.double(), wk.double()), conv64(x.double().abs(), wk.double().abs())
    if not flip:
        ref = ref + b.double()
        ref, mag = torch.where(ref > 0, ref, ref / 64), mag + b.double().abs()
    bound = (27 * ci + 2) * 2.0 ** -24 * mag
    try:
        for fold in (True, False):
            nn.mach_nn_set_conv_fold(fold, 4)
            y32 = torch.full(shape + (co,), 7.0, device="cuda")
            y16 = torch.full(shape + (co,), 7.0, device="cuda", dtype=torch.bfloat16)
            nn.mach_nn_conv3d_tc(x, pk, co, None if flip else b, y16, y32, act=not flip, flip=flip)
            assert nn.mach_nn_device_status() == 0
            assert bool(((y32.double() - ref).abs() <= bound).all()), fold
            assert torch.equal(y16, y32.to(torch.bfloat16)), fold
    finally:
        nn.mach_nn_set_conv_fold(True, 4)
