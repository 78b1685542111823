"""Device-memory caps under which a call has to run: buffers that only make it faster are left out there.

The caps are those of the buffers that the CUDA-core kernels need (T_ii batch and OSVs, pair store, one preconditioner's work
area a CTA, amplitudes, one relaxed-gradient work area a CTA and the eigenvectors of T_ii), a few MiB above the
sizes at which the first of them does not fit; results are those of a context without a cap.
"""
import numpy as np
import pytest

import synth

torch = pytest.importorskip("torch")
pytestmark = pytest.mark.gpu

DEV = "cuda:0"


def _t(x):
    return torch.tensor(np.ascontiguousarray(x), dtype=torch.float64, device=DEV)


def _run(dims, l_osv, call, **kw):
    from paper_2603_16575_gb300 import Context
    s = synth.make_system(*dims, seed=4, lam=1.5)
    ctx = Context(0, **kw)
    ctx.build_osv(_t(s.f_occ), _t(s.e_vir), l_osv, env=_t(s.env), seed=s.seed, n_aux=s.n_aux, r_occ=s.r_occ)
    out = call(ctx)
    again = call(ctx)
    ctx.close()
    return [np.asarray(x.cpu() if torch.is_tensor(x) else x) for x in (*out, *again)]


def _solve(ctx):
    E, pe, _ = ctx.solve(range(min(4, ctx.n_occ)))
    return E, pe


def _relaxed(ctx):
    return ctx.energy_grad_relaxed(7.0, 6.0)[:4]


@pytest.mark.parametrize("dims,l_osv,call,cap", [
    ((6, 64, 150), 1e-4, _solve, 10), ((8, 120, 300), 1e-4, _solve, 30), ((1, 200, 220), 0.0, _solve, 6),
    ((6, 64, 150), 1e-4, _relaxed, 160), ((6, 64, 150), 1e-4, _relaxed, 200), ((1, 200, 220), 0.0, _relaxed, 14)],
    ids=lambda x: getattr(x, "__name__", str(x)))
def test_calls_within_a_cap(dims, l_osv, call, cap):
    free, capped = _run(dims, l_osv, call), _run(dims, l_osv, call, mem_cap_mib=cap)
    for a, b in zip(free, capped):
        assert np.abs(a - b).max() <= 1e-9 * np.abs(a).max()
