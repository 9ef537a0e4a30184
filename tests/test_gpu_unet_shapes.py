"""The U-Net's kernels at cube sides whose tiles are ragged on every level: the
persistent convolutions' tiles (16 x 8 x up to 8), split outputs and up-sampled
inputs, the weight gradients' voxel tiles (4 x 4 x 8), against the CPU oracle; and
an input that is not 16-byte aligned against the same input that is.

Tolerances: those of the 16-cube parity test (2 % of the output and of the loss, 5 %
of a layer's gradient, 8 % where it sums over 16 voxels or so: BF16 rounding flips
that do not average out), and 20 % where it sums over 8."""
import numpy as np
import pytest

from oracle import unet as ounet
from tests.gpu_util import require_gpu

pytestmark = pytest.mark.gpu

LEVEL = (0, 0, 1, 1, 2, 2, 3, 3, 2, 2, 1, 1, 0, 0, 0)


@pytest.fixture(scope="module")
def torch():
    return require_gpu()


def _batch(S, B, seed):
    rng = np.random.default_rng(seed)
    x, y, z = np.meshgrid(*[np.arange(S) - S // 2] * 3, indexing="ij")
    mask = x * x + y * y + z * z <= (S / 2) ** 2
    inp, tgt = np.zeros((B, S, S, S, 3), np.float32), np.zeros((B, S, S, S), np.float32)
    for b in range(B):
        sh = rng.uniform(-1, 1, 3)
        q = (x - sh[0]) ** 2 + (y - sh[1]) ** 2 + (z - sh[2]) ** 2
        inp[b, ..., 0] = np.exp(-q * rng.uniform(4, 8) / S ** 2) * mask
        inp[b, ..., 1] = 5.0 / (np.sqrt(q) + 1.0) * ~mask
        inp[b, ..., 2] = mask
        tgt[b] = 5.0 / (np.sqrt(q) + 1.0) * mask
    return inp, tgt


@pytest.mark.parametrize("S,B", [(16, 1), (24, 1), (32, 2)])
def test_ragged_sides_match_the_oracle(torch, S, B):
    from paper_1911_10630_gb300.exx import GuessNet
    inp, tgt = _batch(S, B, S)
    p = ounet.init_params(12) + np.random.default_rng(13).normal(0, 0.02, ounet.param_count()).astype(np.float32)
    net = GuessNet(S, B)
    net.set_params(p)
    di, dt = torch.from_numpy(inp).cuda(), torch.from_numpy(tgt).cuda()
    out = torch.empty((B, S, S, S), dtype=torch.float32, device="cuda")
    net.forward(di, out, B)
    ref, _ = ounet.forward(p, inp, bf16=True)
    assert np.linalg.norm(out.cpu().numpy() - ref) <= 2e-2 * np.linalg.norm(ref)
    odd = torch.empty(di.numel() + 1, dtype=torch.float32, device="cuda")[1:].view(di.shape).copy_(di)
    out2 = torch.empty_like(out)
    net.forward(odd, out2, B)
    assert torch.equal(out, out2)
    loss, g = net.gradient(di, dt, B)
    rloss, rg = ounet.loss_and_gradient(p, inp, tgt, bf16=True)
    assert abs(loss - rloss) <= 2e-2 * abs(rloss)
    offs = np.concatenate([[0], np.cumsum(ounet.param_sizes())])
    for l, level in enumerate(LEVEL):
        voxels = B * (S >> level) ** 3
        tol = 5e-2 if voxels > 32 else 8e-2 if voxels > 10 else 0.2
        a, b = g[offs[l]:offs[l + 1]], rg[offs[l]:offs[l + 1]]
        assert np.linalg.norm(a - b) <= tol * np.linalg.norm(b), (l, np.linalg.norm(a - b) / np.linalg.norm(b))
    net.close()
