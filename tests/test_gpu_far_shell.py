"""The shell beyond the stencil's reach is evaluated in FP32 from coefficients and row
radii formed in FP64: the wide form of the plain FP64 CG and of the marching kernel is
no further from the FP64 oracle than the general kernel's row form, whose operations on
a point are the same (a few coefficients round the other way: 2 %)."""
import numpy as np
import pytest

import oracle
from paper_1911_10630_gb300 import synth
from tests.gpu_util import require_gpu, run_gpu

pytestmark = pytest.mark.gpu


@pytest.fixture(scope="module")
def torch():
    return require_gpu()


@pytest.mark.parametrize("r,extra,aniso", [(8, 6, 0), (12, 5, 1), (16, 8, 0), (24, 8, 1)])
def test_far_shell_error(torch, r, extra, aniso):
    rm = r + extra
    g = 2 * rm + 3
    w = synth.tiny(seed=r, n=3, npts=g, length=0.195 * g, r_pe=r, r_me=rm, tol=1e-9, min_sep=0.3)
    if aniso:
        w.grid = np.array([g, g + 3, g + 1])
        w.cell = np.array([0.195 * g, 0.2 * g, 0.19 * g])
    phi = w.orbitals()
    outs = [run_gpu(w, phi, torch=torch, **kw) for kw in
            (dict(precision=0, preconditioner=1), dict(precision=0), dict(precision=1, preconditioner=1))]
    pairs = outs[0]["pairs"]
    err = np.zeros(3)
    for k in range(len(pairs["i"])):
        ref = oracle.pair_solve(w.cell, w.grid, phi, int(pairs["i"][k]), int(pairs["j"][k]), pairs["g"][k], r, rm,
                                tol=1e-9)
        far = np.zeros(len(ref["off"]), bool)
        far[ref["n_pe"]:] = (ref["off"][ref["n_pe"]:] ** 2).sum(1) > (r + 3) ** 2  # no leg of the stencil reaches these
        for m, out in enumerate(outs):
            v = out["ex"].debug_pair(out["dphi"], k)["v"]
            err[m] += np.sum((v[far] - ref["v"][far]) ** 2) / np.sum(ref["v"][far] ** 2)
    err = np.sqrt(err / len(pairs["i"]))
    print(err)
    assert 0 < err[0] < 1e-6
    assert err[1] <= 1.02 * err[0] and err[2] <= 1.02 * err[0], err
