"""The FP64 form with equal and close virtual levels.

The amplitude iterations and the adjoint of the FP64 form take the polished pair bases as orthonormal and F as
diagonal in them, so groups of virtual levels that are equal, or as close as the rounding of the first (FP32)
diagonalisation and below, have to come out as well as separate ones: energies to 1e-9 Eh of the closed form and of
the oracle (as everywhere in the FP64 form), 1e-11 of their size, and the same bits from run to run.
"""
import dataclasses

import numpy as np
import pytest

import oracle
import synth

torch = pytest.importorskip("torch")
pytestmark = pytest.mark.gpu

DEV = "cuda:0"


def _t(x):
    return torch.tensor(np.ascontiguousarray(x), dtype=torch.float64, device=DEV)


def _levels(n_vir, kind):
    """("groups", k): equal groups of k; ("cluster", k, width): k levels within width, the rest separate;
    ("range", top): levels from 0.1 to top, most of them low; ("signs",): two levels of either sign."""
    g = np.random.default_rng(n_vir)
    e = 0.1 + 4.9 * g.random(n_vir)
    if kind[0] == "groups":
        e = np.repeat(e, kind[1])[:n_vir]
    elif kind[0] == "cluster":
        e[:kind[1]] = 1.7 + kind[2] * g.random(kind[1])
    elif kind[0] == "range":
        e[-(n_vir // 4):] = 10.0 ** (np.log10(kind[1]) * g.random(n_vir // 4))
    else:
        e = np.where(g.random(n_vir) < 0.5, 0.4, -0.1)
    return g.permutation(e)


def _system(n_occ, n_vir, n_aux, kind, **kw):
    s = synth.make_system(n_occ, n_vir, n_aux, seed=n_vir, **kw)
    return dataclasses.replace(s, e_vir=_levels(n_vir, kind))


def _ctx(s, l_osv):
    from paper_2603_16575_gb300 import Context
    ctx = Context(0)
    k = ctx.build_osv(_t(s.f_occ), _t(s.e_vir), l_osv, env=_t(s.env), seed=s.seed, n_aux=s.n_aux, r_occ=s.r_occ)
    return ctx, k


KINDS = ([("groups", k) for k in (2, 3, 8, 40)] + [("cluster", k, w) for k in (12, 40) for w in
         (0.0, 1e-12, 1e-10, 1e-8, 1e-6, 1e-5, 1e-4)] + [("range", 1e2), ("range", 1e4), ("signs",)])


@pytest.mark.parametrize("kind", KINDS, ids=str)
def test_untruncated_solve_equals_the_closed_form(kind):
    s = _system(3, 60, 130, kind, lam=3.0)
    ref = oracle.canonical_mp2_energy(s.B_block, 3, s.f_occ, s.e_vir)
    got = []
    for _ in range(2):
        ctx, _ = _ctx(s, 0.0)
        E, pe, _ = ctx.solve(range(3))
        got.append((E, pe.tobytes()))
        ctx.close()
    assert abs(got[0][0] - ref) < min(1e-9, 1e-11 * abs(ref))
    assert got[0] == got[1]


@pytest.mark.parametrize("kind", [("groups", 2), ("groups", 8), ("cluster", 30, 1e-12), ("cluster", 30, 1e-8),
                                  ("cluster", 30, 1e-6), ("cluster", 30, 1e-4)], ids=str)
def test_truncated_fragments_match_the_oracle(kind):
    s = _system(5, 50, 110, kind, lam=1.5, f_off=3e-2)
    ctx, k = _ctx(s, 1e-4)
    E, _ = ctx.mbe3_energy(6.0, 5.0, "fp64")
    e = ctx.fragment_results()[2]
    o = oracle.OSVSystem(s.B_block, 5, s.e_vir, s.f_occ, l_osv=1e-4)
    assert [q.shape[1] for q in o.Q] == list(k)
    E_ref, per = o.mbe3_energy(s.r_occ, 6.0, 5.0)
    assert abs(E - E_ref) < 1e-9
    assert max(abs(a - b[2]) for a, b in zip(e, per)) < 1e-11
    ctx.close()


@pytest.mark.parametrize("kind", [("groups", 4), ("cluster", 24, 1e-8)], ids=str)
def test_gradient_matches_the_oracle(kind):
    s = _system(5, 40, 80, kind, lam=1.5, f_off=3e-2)
    ctx, _ = _ctx(s, 1e-3)
    E, dB, df, de, _ = ctx.energy_grad(4.5, 4.0)
    o = oracle.OSVSystem(s.B_block, 5, s.e_vir, s.f_occ, l_osv=1e-3)
    E_ref, dB_ref, de_ref, df_ref = oracle.mbe3_energy_gradient(o, s.r_occ, 4.5, 4.0, 40, 80)
    assert abs(E - E_ref) < 1e-9
    for g, r in ((dB, dB_ref), (df, df_ref), (de, de_ref)):
        assert np.abs(g.cpu().numpy() - r).max() < 1e-8 * np.abs(r).max()
    ctx.close()
