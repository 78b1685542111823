"""The whole-GPU localization runs the sequence of rotations of Algorithm 2 in steps of disjoint
pairs; against the oracle's one-by-one sequence at sizes where the steps differ: one and two
orbitals, odd and even counts, more atoms than orbitals, charge matrices in shared memory and
(from 160 orbitals on) in global memory."""
import numpy as np
import pytest

import oracle
import synth

torch = pytest.importorskip("torch")
pytestmark = pytest.mark.gpu


def _both(C, ao, l_loc=1e-8):
    from paper_2603_16575_gb300 import Context
    ref = oracle.pm_localize(C, ao, l_loc=l_loc, max_sweeps=200)
    ctx = Context(0)
    U, L, sweeps = ctx.localize_pm(torch.tensor(C, dtype=torch.float64, device="cuda:0"), ao, l_loc=l_loc, max_sweeps=200)
    ctx.close()
    return ref, U.cpu().numpy(), L, sweeps


@pytest.mark.parametrize("n", [1, 2, 3, 7, 25, 64, 161])
def test_steps_of_disjoint_pairs_follow_the_sequence(n):
    ls = synth.make_loc_system(n, seed=11 + n)
    ref, U, L, sweeps = _both(np.ascontiguousarray(ls.C), ls.atom_ao, 1e-6)
    assert sweeps == ref.sweeps
    assert abs(L - ref.L) <= 1e-11 * max(1.0, ref.L)
    # the same rotations up to rounding: errors ~ eps per rotation and sweep
    assert np.abs(U - ref.U).max() < 1e-9


def test_more_atoms_than_orbitals_and_uneven_atoms():
    rng = np.random.default_rng(5)
    ao = np.array([0, 1, 4, 4, 9, 15, 17, 30, 41, 42, 60], dtype=np.int32)     # one atom without functions
    C = np.ascontiguousarray(np.linalg.qr(rng.standard_normal((60, 7)))[0])
    ref, U, L, sweeps = _both(C, ao, 1e-7)
    assert sweeps == ref.sweeps and abs(L - ref.L) < 1e-11 and np.abs(U - ref.U).max() < 1e-9
