"""The implicit QR of the relaxed gradient runs on a stream of its own beside the exchange and fragment parts.

Every sum has a fixed order, so a missing wait shows as a difference: two contexts on two streams, driven by two
threads at once, give the bits of a context alone, with virtual spaces at the limits of the eigen-solver (16 / 17
and the last order in shared memory) and one to three orbitals a fragment.
"""
import threading

import numpy as np
import pytest

import synth

torch = pytest.importorskip("torch")
pytestmark = pytest.mark.gpu

DEV = "cuda:0"


def _t(x):
    return torch.tensor(np.ascontiguousarray(x), dtype=torch.float64, device=DEV)


def _run(stream, s, reps, out):
    from paper_2603_16575_gb300 import Context
    with torch.cuda.stream(stream):
        ctx = Context(0, stream=stream)
        ctx.build_osv(_t(s.f_occ), _t(s.e_vir), 1e-3, env=_t(s.env), seed=s.seed, n_aux=s.n_aux, r_occ=s.r_occ)
        for _ in range(reps):
            E, dB, df, de, st, gap = ctx.energy_grad_relaxed(4.5, 3.8)
            assert st["n_unconverged"] == 0
            out.append((E, gap, dB.clone(), df.clone(), de.clone()))
        stream.synchronize()
        ctx.close()


@pytest.mark.parametrize("n,nv,nx", [(1, 40, 60), (2, 16, 40), (3, 17, 40), (9, 64, 90), (6, 160, 200), (5, 161, 200)])
def test_relaxed_overlap_two_streams(n, nv, nx):
    s = synth.make_system(n, nv, nx, seed=n, lam=1.2, f_off=3e-2)
    alone, a, b = [], [], []
    _run(torch.cuda.Stream(), s, 1, alone)
    th = [threading.Thread(target=_run, args=(torch.cuda.Stream(), s, 3, o)) for o in (a, b)]
    for x in th:
        x.start()
    for x in th:
        x.join()
    assert len(a) == 3 and len(b) == 3
    for r in a + b:
        assert r[:2] == alone[0][:2]
        assert all(torch.equal(x, y) for x, y in zip(r[2:], alone[0][2:]))
