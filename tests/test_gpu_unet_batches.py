"""A network used with fewer lattices than it was made for.

Its workspaces are sized once, for the largest batch; a smaller batch can cut the
weight gradient's pixels into more splits than the largest does (64 x 64 lattices, 10
against 8: 10 and 16 splits of the 256 -> 256 layer), and gives the bits of a
network made for it.
"""
import pytest
import torch

from paper_1901_11350_gb300 import inputs as I
from paper_1901_11350_gb300 import unet as UN

pytestmark = pytest.mark.gpu


@pytest.mark.parametrize("L,batch_max,batch", [(64, 10, 8), (64, 18, 14), (32, 40, 32)])
@pytest.mark.parametrize("kernel", ["mma", "tcgen05", "tcgen05_halo"])
def test_smaller_batch_gives_the_bits_of_its_own_network(L, batch_max, batch, kernel):
    old = UN.conv_kernel()
    UN.set_conv_kernel(kernel)
    try:
        gen = torch.Generator(device="cuda").manual_seed(5)
        x = torch.randn((batch, L * L, 4), generator=gen, device="cuda")
        x[..., 3] = 0
        x = x / x.norm(dim=-1, keepdim=True)
        f = torch.rand((batch, 4), generator=gen, device="cuda")
        out = []
        for most in (batch_max, batch):
            net = UN.UNet(L, most, I.unet_init(2))
            grad = torch.empty(net.n_params, device="cuda")
            out.append((net.loss_grad(x, f, x.roll(1, 1), grad).item(), grad, net.predict(x, f)))
        assert out[0][0] == out[1][0]
        assert torch.equal(out[0][1], out[1][1]) and torch.equal(out[0][2], out[1][2])
    finally:
        UN.set_conv_kernel(old)
