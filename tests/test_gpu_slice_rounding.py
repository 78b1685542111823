"""Rounding of the mixed form's digits (five slices, 39 bits) at the upper end of a chunk's scale.

A value just below a power of two rounds up to it, the largest magnitude the digits can hold.  Such values lead
their rows here: entries of B one and a few thousand roundings below a power of two, and the components of
orbital vectors that lie on one virtual up to tiny admixtures.  Tolerance: the slices keep 2^-39 of a row's
largest element in every product, so eigenvalues and energies agree to a few 2^-38 of their size; 1e-9
leaves a factor of a hundred and is far from a wrong sign.
"""
import numpy as np
import pytest

import synth

torch = pytest.importorskip("torch")
pytestmark = pytest.mark.gpu

DEV = "cuda:0"


def _run(B, s, l_osv, prec):
    from paper_2603_16575_gb300 import Context
    f, e = (torch.tensor(x, dtype=torch.float64, device=DEV) for x in (s.f_occ, s.e_vir))
    ctx = Context(0, osv_prec=prec)
    k = ctx.build_osv(f, e, l_osv, B=B, r_occ=s.r_occ)
    w = [ctx.get_osv(i)[1] for i in range(s.n_occ)]
    E, _ = ctx.mbe3_energy(50.0, 50.0, prec)
    per = ctx.fragment_results()[2].copy()
    ctx.close()
    return list(k), w, E, per


def _compare(B, s, l_osv):
    k64, w64, E64, per64 = _run(B, s, l_osv, "fp64")
    k, w, E, per = _run(B, s, l_osv, "mixed")
    assert k == k64
    for a, b in zip(w, w64):
        assert (a - b).abs().max() <= 1e-9 * b.max()
    assert abs(E - E64) <= 1e-9 * abs(E64)
    assert np.abs(per - per64).max() <= 1e-9 * np.abs(per64).max()


@pytest.mark.parametrize("below", [2.0 ** -53, 2.0 ** -41, 2.0 ** -39, 0.0])
@pytest.mark.parametrize("sign", [1.0, -1.0])
@pytest.mark.parametrize("scale", [1.0, 2.0 ** -4])
def test_entries_of_b_below_a_power_of_two(below, sign, scale):
    s = synth.make_system(3, 24, 300, seed=6, lam=50.0)
    g = np.random.default_rng(2)
    B = 0.02 * g.standard_normal((3, 24, 300))
    lead = g.integers(0, 300, size=(3, 24))
    np.put_along_axis(B, lead[:, :, None], sign * (1.0 - below), axis=2)     # the largest of its row and chunk
    _compare(torch.tensor(scale * B, device=DEV), s, 0.0)


@pytest.mark.parametrize("mix", [1e-7, 1e-6, 0.0])
def test_vectors_on_one_virtual(mix):
    # every virtual has auxiliary functions of its own, the others meet them only by mix: components 1 - mix^2
    n, v = 3, 20
    s = synth.make_system(n, v, 4 * v, seed=8, lam=50.0)
    g = np.random.default_rng(3)
    B = mix * g.standard_normal((n, v, 4 * v))
    for a in range(v):
        B[:, a, 4 * a:4 * a + 4] = (0.02 + 0.03 * a) * g.standard_normal((n, 4))
    _compare(torch.tensor(B, device=DEV), s, 1e-5)
