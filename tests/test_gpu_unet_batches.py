"""Batch sizes around the packing kernel's groups of four volumes, and far above: every volume of a
batch comes out as it does alone."""
import pytest
import torch

from paper_2604_06257_gb300 import nn

pytestmark = pytest.mark.gpu


@pytest.mark.parametrize("coords", [False, True])
@pytest.mark.parametrize("N", [1, 2, 3, 4, 5, 7, 8, 9, 33, 64])
def test_volumes_of_a_batch_come_out_as_alone(N, coords):
    nx, ny, nz = 10, 14, 6
    gen = torch.Generator(device="cuda").manual_seed(N)
    x = torch.view_as_complex(torch.randn((nx * ny * nz, N, 2), device="cuda", generator=gen))
    x = x * torch.linspace(0.5, 20.0, N, device="cuda")          # volumes of different size
    with nn.UNet(nx, ny, nz, N, levels=2, seed=1, inference_only=True, coords=coords) as net:
        p = torch.randn(net.n_params, generator=torch.Generator().manual_seed(3)) * 0.05
        net.set_params(p.numpy())
        net.set_gain(0.7)
        y = net.forward(x)
    with nn.UNet(nx, ny, nz, 1, levels=2, seed=1, inference_only=True, coords=coords) as one:
        one.set_params(p.numpy())
        one.set_gain(0.7)
        for n in range(N):
            want = one.forward(x[:, n:n + 1].contiguous())
            torch.cuda.synchronize()
            assert torch.equal(y[:, n:n + 1], want), n
