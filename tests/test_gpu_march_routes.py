"""Which kernel takes a ball: the FP32 multigrid CG marches balls from R_PE 8 to 32 whose
hierarchy is steady (from 14 with 512 threads asked for, none with 1024), in CTAs of 128, 256 or 512 threads (four, two, one per SM; the
largest ball's class at least 256), and leaves the others to the general kernel (six CTAs
per SM with one ball, five with several). grid_ctas and threads tell them apart. Then
calls of all classes at once in which every slot takes several pairs of different balls,
against the general FP64 kernel: both solve to a relative residual of 1e-10, which is
held elsewhere to 1e-8 of every pair's energy and 1e-6 of the largest |D_xx| against the
exact solution; two such results differ by twice the first at most."""
import numpy as np
import pytest

from paper_1911_10630_gb300 import synth
from tests.gpu_util import D_GATE_MAXREL, d_maxrel, require_gpu, run_gpu

pytestmark = pytest.mark.gpu

GENERAL = {9, 13, 17, 18, 19, 21, 25, 26, 27, 29, 33, 34, 35}


@pytest.fixture(scope="module")
def torch():
    return require_gpu()


def _init(r, **kw):
    from paper_1911_10630_gb300.exx import Exx
    g = 2 * (r + 4) + 3
    ex = Exx([0.195 * g] * 3, [g] * 3, float("inf"), r, r + 4, precision=1, preconditioner=1, **kw)
    s = ex.stats()
    ex.close()
    return s["threads"], s["grid_ctas"]


@pytest.mark.parametrize("r", range(1, 38))
def test_the_kernel_of_a_ball(torch, r):
    sms = torch.cuda.get_device_properties(0).multi_processor_count
    if r < 8 or r > 32 or r in GENERAL:
        assert _init(r) == (256, 6 * sms)
    elif r <= 24:
        assert _init(r) == (256, 2 * sms)
    else:
        assert _init(r) == (512, sms)
    if 8 <= r <= 16 and r not in GENERAL:  # CTA sizes asked for
        assert _init(r, threads=512) == ((512, sms) if r >= 14 else (512, 2 * sms))
        assert _init(r, threads=1024) == (1024, sms)
        assert _init(r, ctas_per_sm=1) == (256, sms)


@pytest.mark.parametrize("per_sm", [0, 1])
def test_all_classes_in_one_call(torch, per_sm):
    sms = torch.cuda.get_device_properties(0).multi_processor_count
    w = synth.tiny(seed=5, n=44, npts=81, length=0.195 * 81, r_pe=28, r_me=38, r_pair=9.0, tol=1e-10, alpha=(0.5, 2.0),
                   min_sep=0.4)
    w.radii_mode = 1
    phi = w.orbitals()
    ref = run_gpu(w, phi, torch=torch, precision=0, preconditioner=1)
    out = run_gpu(w, phi, torch=torch, precision=1, preconditioner=1, ctas_per_sm=per_sm)
    s, radii = out["stats"], out["pairs"]["radii"][:, 0]
    # 512, 256 and 128 threads, and the general kernel
    assert s["threads"] == 512 and s["grid_ctas"] == (4 if per_sm else 1 + 2 + 4 + 5) * sms
    count = {k: int(np.sum([f(r) for r in radii])) for k, f in
             dict(general=lambda r: r in GENERAL, large=lambda r: r not in GENERAL and r > 24,
                  small=lambda r: r not in GENERAL and r <= 16).items()}
    assert min(count.values()) > 0 and len(set(radii)) > 8, count
    assert len(radii) > 4 * sms if per_sm else len(radii) > 300
    assert s["n_nonconv"] == 0 and ref["stats"]["n_nonconv"] == 0
    np.testing.assert_allclose(out["pairs"]["e_pair"], ref["pairs"]["e_pair"], rtol=2e-8, atol=1e-12)
    assert d_maxrel(out["D"], ref["D"]) <= D_GATE_MAXREL
    # the same pairs on other slots, after other balls
    cen, al = (torch.from_numpy(np.ascontiguousarray(v)).cuda() for v in (w.centers, w.alphas))
    D = torch.empty_like(out["dphi"])
    for _ in range(2):
        out["ex"].compute(out["dphi"], cen, D, alphas=al)
        np.testing.assert_array_equal(out["ex"].pairs()["e_pair"], out["pairs"]["e_pair"])
    out["ex"].close()
