"""The two diagonalisations of the pair preconditioner (FP32 Jacobi for few pairs, implicit QR for many), both
polished to FP64, and Cholesky against the eigen-decomposition of S for dependent pair spaces.

X^T S X = 1 and X^T F X = diag(e~) hold to the rounding of FP64 sums with X: m^2 products of at most
max|X|^2, so 8 m^2 2^-53 max|X|^2 (times the largest virtual energy for F).
"""
import numpy as np
import pytest

import synth

torch = pytest.importorskip("torch")
pytestmark = pytest.mark.gpu

DEV = "cuda:0"
EPS = 2.0 ** -53


def _t(x):
    return torch.tensor(np.ascontiguousarray(x), dtype=torch.float64, device=DEV)


def _check(ctx, i, j, e_max):
    X, et = ctx.get_precond(i, j)
    _, S, F = ctx.get_pair_blocks(i, j)
    m, r = X.shape
    tol = 8 * m * m * EPS * max(1.0, float(X.abs().max()) ** 2)
    assert (X.T @ S @ X - torch.eye(r, dtype=X.dtype, device=DEV)).abs().max() <= tol
    assert (X.T @ F @ X - torch.diag(et)).abs().max() <= tol * e_max
    return et, tol


# 36 orbitals of 46 OSVs: 666 pairs of order 92 take the QR, three of them alone the Jacobi rotations
def test_many_and_few_pairs_give_the_same_basis():
    from paper_2603_16575_gb300 import Context
    s = synth.make_system(36, 120, 46, seed=5, lam=50.0)
    e_max = float(np.abs(s.e_vir).max())
    got = []
    some = [(0, 1), (4, 30), (17, 17)]
    for pairs in ([(i, j) for i in range(36) for j in range(i, 36)], some):
        ctx = Context(0)
        k = ctx.build_osv(_t(s.f_occ), _t(s.e_vir), 1e-12, env=_t(s.env), seed=s.seed, n_aux=s.n_aux, r_occ=s.r_occ)
        assert min(k) >= 44
        ctx.pair_integrals(pairs, "fp64")
        got.append([_check(ctx, i, j, e_max) for i, j in some])
        ctx.close()
    for (a, tol), (b, _) in zip(*got):
        assert (a.sort().values - b.sort().values).abs().max() <= 2 * tol * e_max


# pair spaces inside the virtual space (independent), filling it and larger than it (dependent)
@pytest.mark.parametrize("n_vir,n_aux", [(40, 12), (40, 20), (40, 33), (24, 40), (70, 34), (70, 36)])
def test_independent_and_dependent_pair_spaces(n_vir, n_aux):
    from paper_2603_16575_gb300 import Context
    s = synth.make_system(3, n_vir, n_aux, seed=n_vir + n_aux, lam=50.0)
    ctx = Context(0)
    ctx.build_osv(_t(s.f_occ), _t(s.e_vir), 1e-12, env=_t(s.env), seed=s.seed, n_aux=s.n_aux, r_occ=s.r_occ)
    ctx.pair_integrals([(0, 1), (1, 2)], "fp64")
    for i, j in ((0, 1), (1, 2), (2, 2)):
        _check(ctx, i, j, float(np.abs(s.e_vir).max()))
        assert ctx.get_precond(i, j)[0].shape[1] <= n_vir
    ctx.close()
