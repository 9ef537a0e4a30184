"""exx_debug_pair re-solves a pair with the kernel and the launch shape of the last call:
its potential gives the call's energy of that pair to rounding, although at a loose
tolerance every kernel stops at another iterate. The last call's stats stay."""
import numpy as np
import pytest

from paper_1911_10630_gb300 import synth
from tests.gpu_util import require_gpu, run_gpu

pytestmark = pytest.mark.gpu


@pytest.fixture(scope="module")
def torch():
    return require_gpu()


MG, FP64 = dict(precision=1, preconditioner=1), dict(precision=0)
CASES = [(8, 0, MG), (16, 0, MG), (24, 0, MG), (28, 0, MG), (17, 0, MG), (25, 12, MG), (20, 12, MG), (16, 0, FP64),
         (12, 0, FP64), (24, 0, FP64), (16, 0, dict(FP64, preconditioner=1))]


@pytest.mark.parametrize("r,r_ns,opts", CASES, ids=["-".join([str(r), str(n)] + [f"{k}{v}" for k, v in o.items()])
                                                    for r, n, o in CASES])
def test_the_debugged_pair_is_the_calls(torch, r, r_ns, opts):
    g = 2 * (r + 4) + 3
    w = synth.tiny(seed=r, n=3, npts=g, length=0.195 * g, r_pe=r, r_me=r + 4, tol=1e-3, min_sep=0.3)
    kw = dict(opts)
    if r_ns:
        kw.update(radii_mode=2, r_pe_nonself=r_ns, r_me_nonself=r_ns + 4)
    out = run_gpu(w, torch=torch, **kw)
    ex, pairs = out["ex"], out["pairs"]
    dv = float(np.prod(np.asarray(w.cell) / np.asarray(w.grid)))
    for k in range(len(pairs["i"])):
        R = int(pairs["radii"][k][0])
        x = np.arange(-R, R + 1)
        n_pe = int((x[:, None, None] ** 2 + x[None, :, None] ** 2 + x[None, None, :] ** 2 <= R * R).sum())
        d = ex.debug_pair(out["dphi"], k)
        e = dv * float(np.dot(d["rho"][:n_pe], d["v"][:n_pe]))
        assert abs(e - pairs["e_pair"][k]) <= 1e-12 * abs(e), k
        assert np.abs(d["b"][:n_pe]).max() > 0
    assert ex.stats() == out["stats"]
    ex.close()
