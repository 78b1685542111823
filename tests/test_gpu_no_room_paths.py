"""The FP64 paths that run without room for the digits: the CUDA-core preconditioner, solver and adjoint.

Few orbitals with large pairs, where the digits of one fragment take more than the work areas of the CUDA-core solver.  The
launches of a repeated call tell which path it took (the CUDA-core solver is one launch for all sweeps, two a sweep for
osvmp2_solve); both must give the same energies and gradients.
"""
import numpy as np
import pytest

import synth

torch = pytest.importorskip("torch")
pytestmark = pytest.mark.gpu

DEV = "cuda:0"


def _t(x):
    return torch.tensor(np.ascontiguousarray(x), dtype=torch.float64, device=DEV)


def _run(dims, call, **kw):
    from paper_2603_16575_gb300 import Context, osvmp2
    s = synth.make_system(*dims, seed=4, lam=1.5)
    ctx = Context(0, **kw)
    ctx.build_osv(_t(s.f_occ), _t(s.e_vir), 0.0, env=_t(s.env), seed=s.seed, n_aux=s.n_aux, r_occ=s.r_occ)
    first = call(ctx)
    before = osvmp2.kernel_launches()
    again = call(ctx)
    n = osvmp2.kernel_launches() - before
    ctx.close()
    return n, [np.asarray(x.cpu() if torch.is_tensor(x) else x) for x in (*first, *again)]


CALLS = {"mbe3": lambda c: (c.mbe3_energy(7.0, 6.0, "fp64")[0], c.fragment_results()[2].copy()),
         "solve": lambda c: c.solve(range(c.n_occ))[:2],
         "grad": lambda c: c.energy_grad(7.0, 6.0, "fp64")[:4],
         "relaxed": lambda c: c.energy_grad_relaxed(7.0, 6.0)[:4]}


@pytest.mark.parametrize("dims,call,cap", [((1, 200, 220), "mbe3", 14), ((1, 200, 220), "mbe3", 60), ((1, 200, 220), "grad", 14),
                                           ((1, 200, 220), "grad", 60), ((1, 200, 220), "relaxed", 60), ((2, 150, 160), "mbe3", 66),
                                           ((2, 150, 160), "solve", 40), ((2, 150, 160), "grad", 66), ((2, 150, 160), "relaxed", 66)])
def test_paths_without_room_give_the_same_results(dims, call, cap):
    usual, free = _run(dims, CALLS[call])
    n, capped = _run(dims, CALLS[call], mem_cap_mib=cap)
    assert n < usual - 4
    for a, b in zip(free, capped):
        assert np.abs(a - b).max() <= 1e-10 * np.abs(a).max()
