"""The FP32 multigrid CG's marching kernel against the general FP64 kernel (same
hierarchy, FP64 throughout) at the sizes where its layout changes: the smallest
balls with a coarse level; odd and even radii; the last ball of 128, 256 and 512
columns and the first beyond (16/20, 24/28, 34/35); balls that
stay on the general kernel in FP32 (9, 13, 17, 21, 25, 33 to 35), alone, few and
many, and beside others; CTA sizes chosen by the caller; two classes of CTA size in one call;
anisotropic ragged grids (FP64 stencil residuals); the integer residual and its
overflow fallback.

Tolerances: both solve to a relative residual of 1e-10, which the multigrid tests
hold to 1e-8 of every pair's energy and 1e-6 of the largest |D_xx| against the
exact solution; two such results differ by twice the first at most."""
import numpy as np
import pytest

from paper_1911_10630_gb300 import synth
from tests.gpu_util import D_GATE_MAXREL, d_maxrel, require_gpu, run_gpu

pytestmark = pytest.mark.gpu


@pytest.fixture(scope="module")
def torch():
    return require_gpu()


# R_PE, R_PE of the non-self pairs (0: the same), anisotropic, options
CASES = [(4, 0, 0, {}), (5, 0, 1, {}), (8, 0, 0, {}), (9, 0, 0, {}), (13, 0, 0, {}), (16, 0, 0, {}), (17, 0, 1, {}),
         (24, 0, 0, {}), (10, 0, 0, {}), (11, 0, 1, {}), (12, 0, 0, {}), (15, 0, 0, {}), (20, 0, 0, {}), (28, 0, 1, {}),
         (31, 0, 0, {}), (32, 0, 0, {}), (30, 21, 0, {}), (21, 12, 0, {}), (25, 0, 0, {}), (33, 0, 0, {}), (34, 0, 0, {}), (35, 0, 0, {}),
         (16, 0, 0, dict(threads=256)), (17, 0, 0, dict(threads=512)), (9, 0, 1, dict(threads=1024)),
         (24, 0, 0, dict(threads=1024)), (25, 12, 0, {}), (18, 13, 1, {}), (16, 5, 0, dict(ctas_per_sm=1)),
         (20, 0, 0, dict(fixed_residual=1)), (20, 12, 0, dict(fixed_residual=2))]


@pytest.mark.parametrize("r,r_ns,aniso,opts", CASES,
                         ids=["-".join([str(r), str(n), "aniso" if a else "iso"] + [f"{k}{v}" for k, v in o.items()])
                              for r, n, a, o in CASES])
def test_marching_multigrid_against_the_fp64_kernel(torch, r, r_ns, aniso, opts):
    n = 2 * (r + 4) + 3
    w = synth.tiny(seed=r, n=4, npts=n, length=0.195 * n, r_pe=r, r_me=r + 4, tol=1e-10, min_sep=0.3)
    if aniso:
        w.grid = np.array([n, n + 3, n + 1])
        w.cell = np.array([0.195 * n, 0.2 * n, 0.19 * n])
    kw = dict(preconditioner=1)
    if r_ns:
        kw.update(radii_mode=2, r_pe_nonself=r_ns, r_me_nonself=r_ns + 4)
    phi = w.orbitals()
    ref = run_gpu(w, phi, torch=torch, precision=0, **kw)
    out = run_gpu(w, phi, torch=torch, precision=1, **kw, **opts)
    assert out["stats"]["n_nonconv"] == 0 and ref["stats"]["n_nonconv"] == 0
    np.testing.assert_allclose(out["pairs"]["e_pair"], ref["pairs"]["e_pair"], rtol=2e-8, atol=1e-12)
    assert d_maxrel(out["D"], ref["D"]) <= D_GATE_MAXREL
