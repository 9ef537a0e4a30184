"""A convolution whose sample has more than 2^31 input elements: its indices are 64-bit.
Its first and last rows equal the convolution of a crop (the same products, added in
the same order: equal bits)."""
import pytest

from tests.gpu_util import require_gpu

pytestmark = pytest.mark.gpu


@pytest.fixture(scope="module")
def torch():
    return require_gpu()


def test_a_sample_of_more_than_2_to_31_elements(torch):
    from paper_1911_10630_gb300 import exx
    D, H, W, C, K = 2, 8192, 8200, 16, 40
    assert D * H * W * C > 2 ** 31
    g = torch.Generator(device="cuda").manual_seed(1)
    x = torch.zeros((1, D, H, W, C), dtype=torch.bfloat16, device="cuda")
    for part in (x[:, :, :K], x[:, :, -K:], x[:, :, H // 2 - K:H // 2]):
        part.copy_(torch.randn(part.shape, generator=g, device="cuda"))
    w = torch.randn((27, C, C), generator=g, device="cuda") * 0.1
    b = torch.randn(C, generator=g, device="cuda")
    y = torch.empty_like(x)
    exx.unet_conv3d(x, w, b, None, y, 1, D, H, W, C, C, 0)
    for lo, hi in ((0, K), (H - K, H), (H // 2 - K, H // 2)):
        xc = x[:, :, lo:hi].contiguous()
        yc = torch.empty_like(xc)
        exx.unet_conv3d(xc, w, b, None, yc, 1, D, hi - lo, W, C, C, 0)
        assert torch.equal(y[:, :, lo:hi], yc), lo  # the rows around each part are zero, as a crop's padding is
        assert yc.float().abs().max() > 0
