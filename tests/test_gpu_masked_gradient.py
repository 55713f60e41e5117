"""Data gradients that leave the convolution already multiplied by the leaky ReLU's derivative
(masks fetched a tile ahead, several tiles per block, ragged tiles): a one-level network's gradients
against the same chain from the layer functions, unmasked convolutions followed by
mach_nn_lrelu_bwd.  Every rounding is the same, so the chains differ by the order of the
weight and bias gradients' atomics alone."""
import numpy as np
import pytest
import torch

from paper_2604_06257_gb300 import nn

pytestmark = pytest.mark.gpu


@pytest.mark.parametrize("c,shape", [(16, (40, 55, 83)), (16, (3, 5, 9)), (32, (31, 41, 57)), (32, (2, 9, 15)), (64, (17, 33, 25))])
def test_one_level_network_equals_its_layers(c, shape):
    nz, ny, nx = shape
    N, V = 2, nz * ny * nx
    gen = torch.Generator(device="cuda").manual_seed(c + nx)
    # inputs of +-1: each volume's RMS is one, exactly
    few = torch.view_as_complex(torch.stack([torch.randint(0, 2, (V, N), device="cuda", generator=gen) * 2.0 - 1.0,
                                             torch.zeros((V, N), device="cuda")], -1))
    many = torch.view_as_complex(torch.randn((V, N, 2), device="cuda", generator=gen))
    loss = torch.zeros(1, device="cuda")
    with nn.UNet(nx, ny, nz, N, levels=1, base_ch=c, seed=5) as net:
        net.set_gain(0.0)
        p = torch.from_numpy(net.params()).cuda()
        net.backward(few, many, loss)
        got = torch.from_numpy(net.grads()).cuda()
    n = 27 * c * c
    w = [p[k * (n + c):k * (n + c) + n].view(27, c, c).contiguous() for k in range(3)]
    b = [p[k * (n + c) + n:(k + 1) * (n + c)].contiguous() for k in range(3)]
    pk = [nn.mach_nn_pack_weights(x, c, c) for x in w]
    x = torch.zeros((N,) + shape + (c,), device="cuda", dtype=torch.bfloat16)
    x[..., :2] = torch.view_as_real(few).permute(1, 0, 2).reshape((N,) + shape + (2,)).to(torch.bfloat16)
    a, e, g_a, g_e, g_o = (torch.zeros_like(x) for _ in range(5))
    o = torch.zeros(x.shape, device="cuda")
    nn.mach_nn_conv3d_tc(x, pk[0][0], c, b[0], a, None, act=True)
    nn.mach_nn_conv3d_tc(a, pk[1][0], c, b[1], e, None, act=True)
    nn.mach_nn_conv3d_tc(e, pk[2][0], c, b[2], None, o)
    err = o[..., :2] - torch.view_as_real(many).permute(1, 0, 2).reshape((N,) + shape + (2,))
    g_o[..., :2] = ((2.0 * err) * torch.tensor(1.0 / np.float32(2 * V * N), device="cuda")).to(torch.bfloat16)
    nn.mach_nn_conv3d_tc(g_o, pk[2][1], c, None, g_e, None, flip=True)
    nn.mach_nn_lrelu_bwd(g_e, e)
    nn.mach_nn_conv3d_tc(g_e, pk[1][1], c, None, g_a, None, flip=True)
    nn.mach_nn_lrelu_bwd(g_a, a)
    want = []
    for xin, g in ((x, g_a), (a, g_e), (e, g_o)):
        dw, db = torch.zeros((27, c, c), device="cuda"), torch.zeros(c, device="cuda")
        nn.mach_nn_conv3d_wgrad(xin, g, dw)
        nn.mach_nn_bias_grad(g, db)
        want += [dw.view(-1), db]
    assert nn.mach_nn_device_status() == 0
    at = 0
    for k, part in enumerate(want):
        mine = got[at:at + part.numel()]
        at += part.numel()
        # float32 sums of up to 456 blocks' atomics in any order: a few units of 2^-24, relative
        # to the terms, which cancel to a few hundredths of their size
        assert float((mine - part).norm()) <= 2e-5 * float(part.norm()) + 1e-12, (k, float((mine - part).norm() / part.norm()))
    assert at == got.numel()
