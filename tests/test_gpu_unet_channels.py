"""Convolutions whose output channels have no even split into slices of 32 or more run
as one slice through one stage; against the CPU oracle, with the tolerances of the other
convolutions (FP32 accumulation of BF16 products, one BF16 rounding of the result)."""
import numpy as np
import pytest

from oracle import unet as ounet
from tests.gpu_util import require_gpu

pytestmark = pytest.mark.gpu


@pytest.fixture(scope="module")
def torch():
    return require_gpu()


@pytest.mark.parametrize("B,D,H,W,cin,cout", [(1, 5, 18, 9, 48, 80), (2, 4, 17, 8, 16, 112), (1, 3, 5, 10, 80, 176),
                                              (1, 6, 16, 8, 32, 208), (1, 1, 33, 20, 32, 96)])
def test_uneven_output_channels(torch, B, D, H, W, cin, cout):
    from paper_1911_10630_gb300 import exx
    rng = np.random.default_rng(cout)
    x = ounet.bf16_round(rng.normal(size=(B, D, H, W, cin)))
    w = rng.normal(0, 0.2, size=(27, cin, cout)).astype(np.float32)
    bias = rng.normal(0, 0.5, size=cout).astype(np.float32)
    ref = np.maximum(ounet.conv3(x, ounet.bf16_round(w), bias.astype(np.float64)), 0)
    dx = torch.from_numpy(np.ascontiguousarray(x, np.float32)).cuda().bfloat16()
    y = torch.empty((B, D, H, W, cout), dtype=torch.bfloat16, device="cuda")
    exx.unet_conv3d(dx, torch.from_numpy(w).cuda(), torch.from_numpy(bias).cuda(), None, y, B, D, H, W, cin, cout, 1)
    out = y.float().cpu().numpy().astype(np.float64)
    scale = np.max(np.abs(ref))
    assert np.max(np.abs(out - ref)) <= 8e-3 * scale + 1e-6
    assert np.linalg.norm(out - ref) <= 4e-3 * np.linalg.norm(ref)
