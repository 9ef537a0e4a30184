"""The general FP32 multigrid kernel's threads per CTA: 256 or, for at most two pairs per
SM and no choice of the caller's, 512 with the same results bit for bit; a caller's
choice is kept, and the stats name what ran."""
import numpy as np
import pytest

from paper_1911_10630_gb300 import synth
from tests.gpu_util import require_gpu, run_gpu

pytestmark = pytest.mark.gpu


@pytest.fixture(scope="module")
def torch():
    return require_gpu()


# R_PE 9, 13, 17: balls that stay on the general kernel; 4 and 40 orbitals: 10 and 820 pairs
@pytest.mark.parametrize("r,n,threads,ran", [(17, 4, 0, 512), (17, 4, 256, 256), (17, 4, 512, 512), (13, 4, 256, 256),
                                             (9, 40, 0, 256), (9, 40, 256, 256)])
def test_threads_of_the_general_kernel(torch, r, n, threads, ran):
    g = 2 * (r + 4) + 3
    w = synth.tiny(seed=r, n=n, npts=g, length=0.195 * g, r_pe=r, r_me=r + 4, tol=1e-9, min_sep=0.05)
    kw = dict(precision=1, preconditioner=1)
    out = run_gpu(w, torch=torch, threads=threads, **kw)
    assert out["stats"]["threads"] == ran
    if threads != 512:
        ref = run_gpu(w, torch=torch, **kw)
        np.testing.assert_array_equal(out["pairs"]["e_pair"], ref["pairs"]["e_pair"])
        np.testing.assert_array_equal(out["pairs"]["iters"], ref["pairs"]["iters"])
