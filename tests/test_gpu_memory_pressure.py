"""FP64 calls after a shortage of device memory.

The digits of the pair bases are given up when a call finds no room; once there is room again the tensor-core solver has
to run again (same launches, same energies), not the CUDA-core one for the rest of the system's life.  The same for
pairs that were built while there was no room for their digits.
"""
import numpy as np
import pytest

import synth

torch = pytest.importorskip("torch")
pytestmark = pytest.mark.gpu

DEV = "cuda:0"


def _t(x):
    return torch.tensor(np.ascontiguousarray(x), dtype=torch.float64, device=DEV)


def _build(ctx, s, l_osv=1e-4):
    return ctx.build_osv(_t(s.f_occ), _t(s.e_vir), l_osv, env=_t(s.env), seed=s.seed, n_aux=s.n_aux, r_occ=s.r_occ)


def _energy(ctx, call):
    from paper_2603_16575_gb300 import osvmp2
    before = osvmp2.kernel_launches()
    E = call(ctx)
    return osvmp2.kernel_launches() - before, E


CALLS = {"mbe3": lambda ctx: ctx.mbe3_energy(7.0, 6.0, "fp64")[0], "solve": lambda ctx: ctx.solve(range(4))[0],
         "grad": lambda ctx: ctx.energy_grad(7.0, 6.0, "fp64")[0]}


@pytest.mark.parametrize("call", CALLS)
def test_digits_given_up_come_back(call):
    from paper_2603_16575_gb300 import Context, osvmp2
    s = synth.make_system(6, 64, 150, seed=4, lam=1.5)
    ctx = Context(0)
    _build(ctx, s)
    _energy(ctx, CALLS[call])
    usual, E = _energy(ctx, CALLS[call])
    ctx.set_opts(mem_cap_mib=1)          # any new block is refused: the digits go
    with pytest.raises(osvmp2.OSVMP2Error) as err:
        ctx.energy_grad_relaxed(7.0, 6.0)
    assert err.value.code == osvmp2.STATUS_CODES["E_NOMEM"]
    ctx.set_opts(mem_cap_mib=0)
    first, E1 = _energy(ctx, CALLS[call])
    again, E2 = _energy(ctx, CALLS[call])
    assert first >= usual and again == usual
    for x in (E1, E2):
        assert abs(x - E) <= 1e-13 * abs(E)
    ctx.close()


def test_pairs_built_without_room_get_their_digits_later():
    from paper_2603_16575_gb300 import Context, osvmp2
    s = synth.make_system(6, 64, 150, seed=4, lam=1.5)
    call = CALLS["solve"]
    ctx = Context(0)
    _build(ctx, s)
    _energy(ctx, call)
    usual, E = _energy(ctx, call)
    ctx.close()
    slow = 0
    for cap in range(8, 24):
        ctx = Context(0, mem_cap_mib=cap)
        try:
            _build(ctx, s)
            _energy(ctx, call)
            n, E1 = _energy(ctx, call)
        except osvmp2.OSVMP2Error as err:
            assert err.code == osvmp2.STATUS_CODES["E_NOMEM"]
            ctx.close()
            continue
        assert abs(E1 - E) <= 1e-12 * abs(E)
        if n < usual:                    # the CUDA-core solver: two launches a sweep
            slow += 1
            ctx.set_opts(mem_cap_mib=0)
            _energy(ctx, call)
            n, E2 = _energy(ctx, call)
            assert n == usual
            assert abs(E2 - E) <= 1e-12 * abs(E)
        ctx.close()
    assert slow > 0
