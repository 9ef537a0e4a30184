"""Orbitals scaled by a power of two: rho and the potentials scale by its square, the
energies by its fourth power and D_xx by its third, exactly. Every FP64 step and the
power-of-two scales of the fixed-point and FP32 copies keep the bits, so the iteration
counts and the pairs' energies are equal to the last bit; D_xx differs by the order of
its atomic adds. The shell beyond the stencil's reach, which only feeds D_xx, has FP32
coefficients in every kernel: D_xx is compared where they lie in FP32's range."""
import numpy as np
import pytest

from paper_1911_10630_gb300 import synth
from tests.gpu_util import d_maxrel, require_gpu, run_gpu

pytestmark = pytest.mark.gpu


@pytest.fixture(scope="module")
def torch():
    return require_gpu()


FP64, MARCH = dict(precision=0), dict(precision=1, preconditioner=1)
CASES = [(r, s, o) for r, s in ((9, 33), (12, 24), (16, 33), (16, -100), (24, 30)) for o in (FP64, MARCH)]
CASES += [(16, 33, dict(precision=0, fixed_residual=1)), (16, 33, dict(precision=1))]


@pytest.mark.parametrize("r,s,opts", CASES, ids=["-".join([str(r), f"2^{s}"] + [f"{k}{v}" for k, v in o.items()])
                                                 for r, s, o in CASES])
def test_powers_of_two_scale_through(torch, r, s, opts):
    g = 2 * (r + 4) + 3
    w = synth.tiny(seed=r, n=4, npts=g, length=0.195 * g, r_pe=r, r_me=r + 4, tol=1e-9, min_sep=0.3)
    phi = w.orbitals()
    ref = run_gpu(w, phi, torch=torch, **opts)
    out = run_gpu(w, np.ldexp(phi, s), torch=torch, **opts)
    assert out["stats"]["n_nonconv"] == 0
    np.testing.assert_array_equal(out["pairs"]["iters"], ref["pairs"]["iters"])
    np.testing.assert_array_equal(np.ldexp(out["pairs"]["e_pair"], -4 * s), ref["pairs"]["e_pair"])
    if abs(s) < 40:
        assert d_maxrel(np.ldexp(out["D"], -3 * s), ref["D"]) <= 1e-12
