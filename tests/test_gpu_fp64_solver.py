"""The FP64 amplitude iterations in the polished preconditioner basis on the tensor cores: pair orders
around the tiles and the scale chunk (columns 64, rows 128, 256), fragments of one to three and of many
orbitals, coefficients that vanish, against the closed form, the oracle and the CUDA-core solver that runs
when the device-memory cap leaves no room for the digits."""
import numpy as np
import pytest

import oracle
import synth

torch = pytest.importorskip("torch")
pytestmark = pytest.mark.gpu

DEV = "cuda:0"


def _t(x):
    return torch.tensor(np.ascontiguousarray(x), dtype=torch.float64, device=DEV)


def _build(ctx, s, l_osv):
    return ctx.build_osv(_t(s.f_occ), _t(s.e_vir), l_osv, env=_t(s.env), seed=s.seed, n_aux=s.n_aux, r_occ=s.r_occ)


@pytest.mark.parametrize("n_occ,n_vir", [(1, 5), (2, 31), (2, 64), (2, 65), (3, 129), (2, 257), (5, 33)])
def test_untruncated_orders_around_the_tiles_equal_the_closed_form(n_occ, n_vir):
    # pair basis order = n_vir; the closed form holds to the rounding of the FP64 energies
    from paper_2603_16575_gb300 import Context
    s = synth.make_system(n_occ, n_vir, 2 * n_vir + 3, seed=n_vir, lam=3.0)
    ctx = Context(0)
    _build(ctx, s, 0.0)
    E, pe, it = ctx.solve(range(n_occ))
    ref = oracle.canonical_mp2_energy(s.B_block, n_occ, s.f_occ, s.e_vir)
    assert abs(E - ref) < 1e-9
    assert np.isclose(pe.sum(), E, rtol=1e-13, atol=0.0)
    ctx.close()


@pytest.mark.parametrize("f_off", [0.0, 3e-2])
def test_fragments_match_the_oracle_with_and_without_couplings(f_off):
    from paper_2603_16575_gb300 import Context
    s = synth.make_system(7, 60, 130, seed=9, lam=1.2, f_off=f_off)
    ctx = Context(0)
    _build(ctx, s, 1e-4)
    E, st = ctx.mbe3_energy(6.0, 5.0, "fp64")
    o = oracle.OSVSystem(s.B_block, s.n_occ, s.e_vir, s.f_occ, l_osv=1e-4)
    E_ref, per = o.mbe3_energy(s.r_occ, 6.0, 5.0)
    _, _, e = ctx.fragment_results()
    assert abs(E - E_ref) < 1e-9
    assert max(abs(a - b[2]) for a, b in zip(e, per)) < 1e-11
    ctx.close()


def test_polished_basis_is_orthonormal_and_diagonal():
    # X^T S X and X^T F X from blocks of FP64 accuracy carry eps |X|^2, X ~ lambda_min(S)^(-1/2)
    from paper_2603_16575_gb300 import Context
    s = synth.make_system(4, 90, 150, seed=3, lam=1.5)
    ctx = Context(0)
    _build(ctx, s, 1e-4)
    ctx.pair_integrals([(0, 1), (2, 3)], "fp64")
    for i, j in ((0, 1), (2, 3), (1, 1)):
        _, S, F = ctx.get_pair_blocks(i, j)
        X, et = ctx.get_precond(i, j)
        tol = 64 * 2.0 ** -53 * float((X * X).sum(0).max())
        assert (X.T @ S @ X - torch.eye(X.shape[1], dtype=torch.float64, device=DEV)).abs().max() < max(tol, 1e-12)
        assert (X.T @ F @ X - torch.diag(et)).abs().max() < max(tol * float(et.abs().max()), 1e-11)
    ctx.close()


def test_memory_cap_runs_the_cuda_core_solver_with_the_same_energies():
    from paper_2603_16575_gb300 import Context, osvmp2
    s = synth.make_system(6, 64, 150, seed=4, lam=1.5)
    ctx = Context(0)
    _build(ctx, s, 1e-4)
    E, _ = ctx.mbe3_energy(7.0, 6.0, "fp64")
    e = ctx.fragment_results()[2]
    launches = osvmp2.kernel_launches()
    ctx.mbe3_energy(7.0, 6.0, "fp64")
    free_launches = osvmp2.kernel_launches() - launches
    ctx.close()
    ran = 0
    for cap in (40, 60, 90, 140, 200, 300):
        c = Context(0, mem_cap_mib=cap)
        try:
            _build(c, s, 1e-4)
            launches = osvmp2.kernel_launches()
            E2, _ = c.mbe3_energy(7.0, 6.0, "fp64")
            ran += 1
        except osvmp2.OSVMP2Error as err:
            assert err.code == osvmp2.STATUS_CODES["E_NOMEM"]
            c.close()
            continue
        assert abs(E2 - E) < 1e-11 * abs(E)
        assert np.abs(c.fragment_results()[2] - e).max() < 1e-11 * np.abs(e).max()
        c.close()
    assert ran > 0 and free_launches > 0
