"""Contexts of different sizes on several host threads at once.

How much dynamic shared memory a kernel may ask for is a property of the process.  The smaller system's launches must not
take it from the larger one's between its call and its launch: all threads have to see the results of a context alone,
with pair orders and virtual spaces that need much and little of it, in both forms, with all and with some OSVs.
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


def _calls(stream, s, repeat, out):
    from paper_2603_16575_gb300 import Context
    try:
        with torch.cuda.stream(stream):
            ctx = Context(0, stream)
            f, e, env = _t(s.f_occ), _t(s.e_vir), _t(s.env)
            stream.synchronize()
            for _ in range(repeat):
                got = []
                for l_osv, precs in ((0.0, ("mixed", "fp64")), (1e-4, ("mixed",))):
                    ctx.build_osv(f, e, l_osv, env=env, seed=s.seed, n_aux=s.n_aux, r_occ=s.r_occ)
                    got += [ctx.mbe3_energy(50.0, 50.0, prec)[0] for prec in precs]
                out.append(got)
            ctx.close()
    except Exception as err:          # seen by the main thread
        out.append(err)


def test_threads_with_systems_of_different_sizes():
    large = synth.make_system(2, 150, 160, seed=3, lam=3.0)
    small = synth.make_system(1, 20, 40, seed=4, lam=3.0)
    alone = []
    for s in (large, small):
        out = []
        _calls(torch.cuda.current_stream(), s, 1, out)
        alone.append(out[0])
    plan = [(large, 60), (small, 600), (small, 600), (large, 60)]
    got = [[] for _ in plan]
    th = [threading.Thread(target=_calls, args=(torch.cuda.Stream(), s, r, o)) for (s, r), o in zip(plan, got)]
    for t in th:
        t.start()
    for t in th:
        t.join()
    for (s, r), out in zip(plan, got):
        for x in out:
            assert not isinstance(x, Exception), x
            assert x == alone[0 if s is large else 1]
