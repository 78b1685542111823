"""Mixed form against the FP64 form, and the pair screening, at the sizes where their tiles can go wrong.

Fragments with pair orders around 32, 64 and 128 (tile widths and heights, k-blocks), virtual and auxiliary counts
around a k-block and a scale chunk (32, 256), one orbital to all three-orbital fragments.  Tolerance: the
overlaps of the pair bases are FP32 (2^-24 an entry) in coupling terms of ~1e-2 of the denominators, the
rest carries 31 bits and more, so a fragment energy is within a few 1e-10 of its value; 1e-8 leaves the
conditioning of the amplitude equations and is far from any indexing mistake.
"""
import numpy as np
import pytest

import synth

torch = pytest.importorskip("torch")
pytestmark = pytest.mark.gpu

DEV = "cuda:0"


def _t(x):
    return torch.tensor(np.ascontiguousarray(x), dtype=torch.float64, device=DEV)


def _ctx(s, l_osv, **kw):
    from paper_2603_16575_gb300 import Context
    ctx = Context(0, **kw)
    ctx.build_osv(_t(s.f_occ), _t(s.e_vir), l_osv, env=_t(s.env), seed=s.seed, n_aux=s.n_aux, r_occ=s.r_occ)
    return ctx


@pytest.mark.parametrize("n_occ,n_vir,n_aux,l_osv", [(1, 17, 31, 1e-4), (3, 31, 33, 1e-5), (5, 33, 64, 1e-6), (4, 66, 255, 1e-7),
                                                     (5, 96, 257, 1e-6), (4, 150, 288, 1e-7), (3, 257, 300, 1e-6)])
def test_mixed_fragment_energies_match_fp64(n_occ, n_vir, n_aux, l_osv):
    s = synth.make_system(n_occ, n_vir, n_aux, seed=60 + n_vir, lam=1.2)
    ctx = _ctx(s, l_osv)
    e = {}
    for prec in ("fp64", "mixed"):
        ctx.mbe3_energy(50.0, 50.0, prec)       # every pair and triple
        e[prec] = ctx.fragment_results()[2].copy()
    ctx.close()
    assert np.abs(e["mixed"] - e["fp64"]).max() <= 1e-8 * np.abs(e["fp64"]).max()


@pytest.mark.parametrize("n_occ,n_vir,l_osv", [(2, 1, 0.0), (3, 33, 0.0), (4, 65, 1e-5), (3, 140, 0.0), (5, 260, 1e-6)])
def test_pair_screening_matches_plain_overlaps(n_occ, n_vir, l_osv):
    s = synth.make_system(n_occ, n_vir, n_vir + 20, seed=11, lam=1.5)
    ctx = _ctx(s, l_osv)
    Q = [ctx.get_osv(i)[0] for i in range(n_occ)]
    s2b = np.asarray(ctx.pair_screening()[0])
    ctx.close()
    for i in range(n_occ):
        for j in range(i + 1, n_occ):
            ref = float(((Q[i].T @ Q[j]) ** 2).sum()) / (Q[i].shape[1] * Q[j].shape[1]) ** 0.5
            # n_vir products of columns of norm 1, n_i n_j squares of at most 1
            assert abs(s2b[i, j] - ref) <= 8 * n_vir * 2.0 ** -53 * max(1.0, ref)
