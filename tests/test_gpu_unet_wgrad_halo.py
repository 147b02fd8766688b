"""The weight and bias gradient on halo tiles (image rows of at least 64 pixels).

Against the FP64 restatement of the convolution's backward pass, with the bound
of test_gpu_unet.py (FP32 sums of P products in any order): bands of 4, 2 and 1
rows, rows that are no multiple of 64, upsampled and concatenated inputs, several
channel tiles; and a wait that runs out.
"""
import numpy as np
import pytest
import torch

from oracle import unet as U
from paper_1901_11350_gb300 import build
from paper_1901_11350_gb300 import unet as UN

pytestmark = pytest.mark.gpu


@pytest.fixture(scope="module", autouse=True)
def _lib():
    if not torch.cuda.is_available():
        pytest.skip("no CUDA device")
    build.build()
    old = UN.conv_kernel()
    UN.set_conv_kernel("tcgen05_halo")
    yield
    UN.set_conv_kernel(old)


def rand_bf(rng, shape):
    t = torch.from_numpy(rng.standard_normal(shape).astype(np.float32)).to(torch.bfloat16)
    return t.cuda(), t.float().numpy().astype(np.float64)


def virtual_input(x0, x1, up0):
    x = U.upsample(x0) if up0 else x0
    return x if x1 is None else np.concatenate([x, x1], axis=-1)


def _check(s0, x0, dzt, dz, s1=None, x1=None, up0=0):
    dW, db = UN.conv3x3_wgrad(s0, dzt, src1=s1, up0=bool(up0))
    x = virtual_input(x0, x1, up0)
    Cout, P = dz.shape[-1], int(np.prod(dz.shape[:3]))
    _, rW, rb = U.conv3x3_backward(x, np.zeros((Cout, 9, x.shape[-1])), dz)
    _, SW, Sb = U.conv3x3_backward(np.abs(x), np.zeros((Cout, 9, x.shape[-1])), np.abs(dz))
    assert np.all(np.abs(dW.cpu().numpy().astype(np.float64) - rW) <= 2 * (P + 1024) * 2.0 ** -24 * SW)
    assert np.all(np.abs(db.cpu().numpy().astype(np.float64) - rb) <= 2 * (P + 1024) * 2.0 ** -24 * Sb)
    return dW, db


@pytest.mark.parametrize("case", [
    (2, 8, 64, 32, 0, 0, 32),
    (1, 6, 128, 32, 0, 0, 64),    # two rows a band
    (2, 5, 64, 64, 0, 0, 64),     # one row a band
    (2, 4, 80, 32, 0, 0, 96),     # three channel tiles of 32, rows of 5 steps
    (1, 8, 64, 64, 1, 32, 32),    # upsampled and concatenated
    (1, 4, 256, 32, 0, 64, 32),
    (3, 12, 128, 96, 0, 0, 128),
])
def test_weight_gradient_on_halo_tiles(case):
    B, H, W, C0, up0, C1, Cout = case
    rng = np.random.default_rng(5 + C0 + Cout + W)
    h0, w0 = (H // 2, W // 2) if up0 else (H, W)
    s0, x0 = rand_bf(rng, (B, h0, w0, C0))
    s1, x1 = rand_bf(rng, (B, H, W, C1)) if C1 else (None, None)
    dzt, dz = rand_bf(rng, (B, H, W, Cout))
    a = _check(s0, x0, dzt, dz, s1, x1, up0)
    b = UN.conv3x3_wgrad(s0, dzt, src1=s1, up0=bool(up0))
    assert torch.equal(a[0], b[0]) and torch.equal(a[1], b[1])
    UN.check_device_error()


def test_a_wait_that_runs_out_is_reported():
    # 32 bands of 8 rows over 25 splits: some CTA waits for its first band's MMAs
    rng = np.random.default_rng(3)
    s0, x0 = rand_bf(rng, (4, 64, 64, 128))
    dzt, dz = rand_bf(rng, (4, 64, 64, 96))
    try:
        UN.set_wait_limit(0)
        UN.conv3x3_wgrad(s0, dzt)
        assert UN.lib().sp_unet_device_error() == -5
    finally:
        UN.set_wait_limit()
    _check(s0, x0, dzt, dz)
    assert UN.lib().sp_unet_device_error() == 0


@pytest.mark.parametrize("shape", [(1, 64, 64, 32, 32), (1, 8, 128, 32, 64), (2, 16, 16, 32, 128)])
def test_outputs_and_masks_on_16_byte_boundaries(shape):
    # 32-byte rows at once where out and mask allow it, two 16-byte ones elsewhere
    B, H, W, Cin, Cout = shape
    rng = np.random.default_rng(9)
    x, _ = rand_bf(rng, (B, H, W, Cin))
    Wt, _ = rand_bf(rng, (Cout, 9, Cin))
    mask, _ = rand_bf(rng, (B, H, W, Cout))
    want = UN.conv3x3_forward(x, Wt, None, relu=False, mask=mask)
    n = want.numel()
    for mo, oo in ((0, 8), (8, 0), (8, 8)):
        m = torch.zeros(n + 16, dtype=torch.bfloat16, device="cuda")
        out = torch.full((n + 16,), 7.0, dtype=torch.bfloat16, device="cuda")
        m[mo:mo + n] = mask.reshape(-1)
        rc = UN.lib().sp_conv3x3_forward(x.data_ptr(), Cin, 0, None, 0, Wt.data_ptr(), None, 0, m.data_ptr() + 2 * mo, B,
                                         H, W, Cout, out.data_ptr() + 2 * oo, torch.cuda.current_stream().cuda_stream)
        assert rc == 0
        assert torch.equal(out[oo:oo + n], want.reshape(-1))
        assert bool(torch.all(out[:oo] == 7.0)) and bool(torch.all(out[oo + n:] == 7.0))
    UN.check_device_error()
