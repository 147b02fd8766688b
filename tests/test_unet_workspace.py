"""The weight gradient's workspace: what the query asks for and what a call takes."""
import ctypes

import numpy as np
import pytest
import torch

from paper_1901_11350_gb300 import build
from paper_1901_11350_gb300 import unet as UN


def _query(*shape):
    f = ctypes.CDLL(build.build()).sp_conv3x3_wgrad_workspace
    f.restype = ctypes.c_longlong
    return f(*shape)


@pytest.mark.parametrize("B,H,W,cin,cout", [(1, 16, 16, 32, 32), (2, 32, 32, 32, 64), (1, 8, 64, 32, 32),
                                            (1, 4, 128, 96, 32)])
def test_workspace_asked_for_is_that_of_the_splits_a_call_can_make(B, H, W, cin, cout):
    # a split takes at least 32 pixels, a part of the bias gradient at least one split's
    splits = B * H * W // 32
    assert 0 < _query(B, H, W, cin, cout) <= splits * (9 * cin + 1) * cout * 4


def _tc_bytes(P, cin, cout):
    """Partials of the kernels that take one tap at a time (152 SMs)."""
    need = 0
    for tc in (0, 1):
        if tc:
            bn = 256 if cout % 256 == 0 else 128 if cout % 128 == 0 else 64 if cout % 64 == 0 else 32
            want = max(1, 152 * {256: 2, 128: 3, 64: 4, 32: 5}[bn] // (-(-9 * cin // 128) * (cout // bn)))
        else:
            want = -(-608 // ((cout // (64 if cout % 64 == 0 else 32)) * 9 * (cin // 32)))
        chunks = P // 32
        per = -(-chunks // max(1, min(want, chunks)))
        pix = max(1024, (-(-P // 304) + 63) // 64 * 64)
        need = max(need, (-(-chunks // per) * 9 * cin + -(-P // pix)) * cout * 4)
    return need


@pytest.mark.gpu
@pytest.mark.parametrize("B,H,W,cin,cout", [(1, 16, 16, 32, 32), (4, 64, 64, 128, 96), (8, 128, 128, 32, 32),
                                            (2, 64, 64, 64, 32)])
def test_workspace_of_the_tap_by_tap_kernels_is_taken(B, H, W, cin, cout):
    # by the default kernel too: where it would like more, with the bits of kernel 1
    rng = np.random.default_rng(3)
    bf = lambda *s: torch.from_numpy(rng.standard_normal(s).astype(np.float32)).to(torch.bfloat16).cuda()  # noqa: E731
    x, dz = bf(B, H, W, cin), bf(B, H, W, cout)
    old, out, size, full = UN.conv_kernel(), [], _tc_bytes(B * H * W, cin, cout), _query(B, H, W, cin, cout)
    try:
        for kernel, room in (("tcgen05", size), ("tcgen05_halo", full), ("tcgen05_halo", size), ("tcgen05_halo", size - 1)):
            UN.set_conv_kernel(kernel)
            ws = torch.zeros(full, dtype=torch.uint8, device="cuda")
            dW, db = torch.empty((cout, 9, cin), device="cuda"), torch.empty(cout, device="cuda")
            rc = UN.lib().sp_conv3x3_wgrad(x.data_ptr(), cin, 0, None, 0, dz.data_ptr(), B, H, W, cout, dW.data_ptr(),
                                           db.data_ptr(), ws.data_ptr(), room, torch.cuda.current_stream().cuda_stream)
            torch.cuda.synchronize()
            assert not ws[room:].any()
            out.append((rc, dW, db))
    finally:
        UN.set_conv_kernel(old)
    assert [r[0] for r in out] == [0, 0, 0, -1]
    ref = out[0] if full > size else out[1]
    assert torch.equal(out[2][1], ref[1]) and torch.equal(out[2][2], ref[2])
