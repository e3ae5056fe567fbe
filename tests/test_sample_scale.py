"""The per-sample input scale at the edges of its split over eight blocks: less than a block's share, odd
counts, rows that four-float loads do not fit, a source off a 16-byte boundary.  Against FP64: one FP32
rounding of the result, the sum and the quotient being FP64 (2^-23 relative)."""
import pytest
import torch

from paper_1608_05238_gb300 import _build
from paper_1608_05238_gb300 import denoise_ops as ops

pytestmark = pytest.mark.gpu


@pytest.fixture(scope="module", autouse=True)
def _lib():
    _build.build()


@pytest.mark.parametrize("offset", [0, 1])
@pytest.mark.parametrize("B,C,H,W", [(1, 1, 1, 1), (2, 3, 1, 7), (3, 2, 4, 8), (1, 5, 31, 33), (2, 1, 64, 130),
                                     (4, 2, 257, 255), (1, 9, 512, 512)])
def test_scale_is_inverse_mean(B, C, H, W, offset):
    g = torch.Generator().manual_seed(B * 1000 + H)
    flat = torch.randn(B * C * H * W + offset, generator=g).cuda()
    x = flat[offset:].view(B, C, H, W)
    scale = torch.empty(B, device="cuda")
    ops.sample_scale(x, scale)
    ref = 1.0 / x[:, 0].double().abs().mean(dim=(1, 2))
    assert ((scale.double() - ref).abs() <= 2.0 ** -23 * ref).all()
