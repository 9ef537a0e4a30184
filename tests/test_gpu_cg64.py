"""The plain FP64 CG's team kernel against the general FP64 kernel (multigrid PCG,
FP64 stencil throughout; plain CG below R_PE 4) at the sizes where its layout
changes: balls of a few pairs of points, fewer than the threads of a team; rows
that start on odd and even z; one band of rows and several; teams of 1, 2, 4 and
8 CTAs; every CTA size; the FP64 stencil (anisotropic grids, or on request); two
balls in one call.

Tolerances: both solve to a relative residual of 1e-10, which is held elsewhere
to 1e-8 of every pair's energy and 1e-6 of the largest |D_xx| against the exact
solution; two such results differ by twice the first at most."""
import numpy as np
import pytest

from paper_1911_10630_gb300 import synth
from tests.gpu_util import D_GATE_MAXREL, d_maxrel, require_gpu, run_gpu

pytestmark = pytest.mark.gpu


@pytest.fixture(scope="module")
def torch():
    return require_gpu()


# R_PE, R_PE of the non-self pairs (0: the same), orbitals, anisotropic, options, CTAs per pair
CASES = [(1, 0, 3, 0, {}, 1), (3, 0, 4, 1, {}, 1), (5, 0, 4, 0, {}, 1), (8, 0, 20, 0, {}, 1), (9, 0, 4, 1, {}, 2),
         (12, 0, 4, 0, {}, 4), (13, 0, 3, 1, {}, 4), (16, 0, 4, 0, {}, 8), (17, 0, 8, 0, {}, 4), (16, 0, 12, 0, {}, 1),
         (16, 0, 10, 0, dict(threads=256), 2), (16, 0, 3, 0, dict(threads=1024), 8), (24, 0, 18, 0, {}, 2),
         (33, 0, 3, 0, {}, 8), (20, 0, 4, 0, dict(fixed_residual=1), 8), (20, 9, 4, 0, {}, 8), (18, 13, 8, 1, {}, 4),
         (16, 5, 20, 0, dict(ctas_per_sm=1), 1), (12, 0, 4, 0, dict(deterministic=1), 4)]


@pytest.mark.parametrize("r,r_ns,n,aniso,opts,team", CASES,
                         ids=["-".join([str(r), str(ns), f"n{n}", "aniso" if a else "iso"] +
                                       [f"{k}{v}" for k, v in o.items()]) for r, ns, n, a, o, _ in CASES])
def test_plain_fp64_teams_against_the_general_kernel(torch, r, r_ns, n, aniso, opts, team):
    g = 2 * (r + 4) + 3
    w = synth.tiny(seed=r, n=n, npts=g, length=0.195 * g, r_pe=r, r_me=r + 4, tol=1e-10, min_sep=0.2)
    if aniso:
        w.grid = np.array([g, g + 3, g + 1])
        w.cell = np.array([0.195 * g, 0.2 * g, 0.19 * g])
    kw = dict(precision=0)
    if r_ns:
        kw.update(radii_mode=2, r_pe_nonself=r_ns, r_me_nonself=r_ns + 4)
    phi = w.orbitals()
    ref = run_gpu(w, phi, torch=torch, preconditioner=1, **kw)
    out = run_gpu(w, phi, torch=torch, **kw, **opts)
    assert out["stats"]["n_nonconv"] == 0 and ref["stats"]["n_nonconv"] == 0
    assert out["stats"]["cluster_size"] == team
    np.testing.assert_allclose(out["pairs"]["e_pair"], ref["pairs"]["e_pair"], rtol=2e-8, atol=1e-12)
    assert d_maxrel(out["D"], ref["D"]) <= D_GATE_MAXREL
