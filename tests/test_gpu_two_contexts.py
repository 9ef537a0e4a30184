"""Contexts of different radii alive at once. A kernel's shared-memory limit belongs to
the function, not to the context: creating one that needs less must not take what
another needs. Each first context is called (eagerly, then through its graph) after the
second exists, and gives what it gives alone. The radii share a launch shape and differ
in shared memory."""
import threading

import numpy as np
import pytest

from paper_1911_10630_gb300 import synth
from tests.gpu_util import require_gpu

pytestmark = pytest.mark.gpu


@pytest.fixture(scope="module")
def torch():
    return require_gpu()


MG, FP64 = dict(precision=1, preconditioner=1), dict(precision=0)
CASES = [(22, 20, MG), (22, 24, MG), (16, 8, dict(MG, threads=256)), (32, 28, MG), (25, 13, MG), (24, 12, FP64),
         (24, 12, dict(FP64, preconditioner=1)), (24, 16, dict(precision=1, autotune=0)),
         (24, 16, dict(MG, solver_kind=2))]


def _run(torch, w, phi, ex):
    d = torch.from_numpy(phi).cuda()
    D = torch.empty_like(d)
    cen = torch.from_numpy(np.ascontiguousarray(w.centers)).cuda()
    out = []
    for _ in range(3):
        ex.compute(d, cen, D)
        out.append(ex.pairs()["e_pair"].copy())
    return out


@pytest.mark.parametrize("big,small,opts", CASES, ids=["-".join([str(b), str(s)] + [f"{k}{v}" for k, v in o.items()])
                                                       for b, s, o in CASES])
def test_a_smaller_context_takes_nothing_from_a_larger(torch, big, small, opts):
    from paper_1911_10630_gb300.exx import Exx

    def make(r):
        g = 2 * (r + 4) + 3
        w = synth.tiny(seed=r, n=3, npts=g, length=0.195 * g, r_pe=r, r_me=r + 4, tol=1e-8, min_sep=0.3)
        return w, w.orbitals(), Exx(w.cell, w.grid, w.r_pair, w.r_pe, w.r_me, w.l_max, w.tol, **opts)

    w, phi, first = make(big)
    w2, phi2, second = make(small)
    a = _run(torch, w, phi, first)
    b = _run(torch, w2, phi2, second)
    second.close()
    first.close()
    _, _, alone = make(big)
    ref = _run(torch, w, phi, alone)
    alone.close()
    for e in a[1:] + ref:
        np.testing.assert_array_equal(e, a[0])
    assert all(np.isfinite(e).all() for e in b)


def test_networks_on_two_threads(torch):
    from oracle import unet as ounet
    from paper_1911_10630_gb300.exx import GuessNet
    p = ounet.init_params(3)
    nets, ins, refs, bad = [], [], [], []
    for S in (16, 48):
        net = GuessNet(S, 2)
        net.set_params(p)
        x = torch.rand((2, S, S, S, 3), generator=torch.Generator().manual_seed(S)).cuda()
        y = torch.empty((2, S, S, S), device="cuda")
        net.forward(x, y, 2)
        nets.append(net)
        ins.append(x)
        refs.append(y.cpu())

    def work(k):
        try:
            st = torch.cuda.Stream()
            with torch.cuda.stream(st):
                y = torch.empty_like(refs[k], device="cuda")
                for _ in range(50):
                    nets[k].forward(ins[k], y, 2)
                    st.synchronize()
                    if not torch.equal(y.cpu(), refs[k]):
                        bad.append(k)
        except Exception as e:  # a refused launch
            bad.append(repr(e))

    ts = [threading.Thread(target=work, args=(k,)) for k in range(2)]
    for t in ts:
        t.start()
    for t in ts:
        t.join()
    for net in nets:
        net.close()
    assert not bad, bad[:3]
