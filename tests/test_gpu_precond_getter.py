"""osvmp2_get_precond hands out the basis that the solver uses, also for dependent pair spaces (larger than the virtual
space), where its coefficients are rewritten to the shortest ones: X, e~ and r belong to the built pair, not to the
options of the moment, U = P X is orthonormal with F diagonal in it, and X has no part along the dependent directions.

Tolerance: products with X carry a few m 2^-53 max|X|, those with S and F twice that with max|X|^2.
"""
import numpy as np
import pytest

import oracle
import synth

torch = pytest.importorskip("torch")
pytestmark = pytest.mark.gpu

DEV = "cuda:0"
EPS = 2.0 ** -53


def _t(x):
    return torch.tensor(np.ascontiguousarray(x), dtype=torch.float64, device=DEV)


# overlaps of the pair that are all 0 or 1 (the last), and angles of every size between
@pytest.mark.parametrize("n_vir,n_aux,l_osv", [(40, 20, 1e-3), (40, 33, 1e-2), (24, 40, 1e-2), (70, 36, 1e-3), (40, 33, 1e-4)])
def test_the_solvers_basis_whatever_the_options(n_vir, n_aux, l_osv):
    from paper_2603_16575_gb300 import Context
    s = synth.make_system(3, n_vir, n_aux, seed=n_vir + n_aux, lam=50.0)
    ctx = Context(0)
    ctx.build_osv(_t(s.f_occ), _t(s.e_vir), l_osv, env=_t(s.env), seed=s.seed, n_aux=s.n_aux, r_occ=s.r_occ)
    ctx.pair_integrals([(0, 1), (1, 2)], "fp64")
    Q = [ctx.get_osv(i)[0] for i in range(3)]
    e = _t(s.e_vir)
    for i, j in ((0, 1), (1, 2), (2, 2)):
        X, et = ctx.get_precond(i, j)
        m, r = X.shape
        P = Q[i] if i == j else torch.cat([Q[i], Q[j]], 1)
        U = P @ X
        big = max(1.0, float(X.abs().max()))
        tol = 8 * m * m * EPS * big ** 2
        assert (U.T @ U - torch.eye(r, dtype=X.dtype, device=DEV)).abs().max() <= tol
        assert (U.T @ (e[:, None] * U) - torch.diag(et)).abs().max() <= tol * float(e.max())
        _, S, F = (x.cpu().numpy() for x in ctx.get_pair_blocks(i, j))
        Xr, er = oracle.preconditioner(S, F, 1e-10)
        assert Xr.shape[1] == r
        assert np.abs(np.sort(et.cpu().numpy()) - np.sort(er)).max() <= tol * float(e.max())
        if r < m:
            w, V = np.linalg.eigh(S)
            assert np.abs(V[:, : m - r].T @ X.cpu().numpy()).max() <= 64 * m * EPS * big ** 2
        ctx.set_opts(tau_s=0.3)            # of later builds
        X2, et2 = ctx.get_precond(i, j)
        ctx.set_opts(tau_s=1e-10)
        assert X2.shape == X.shape and torch.equal(X2, X) and torch.equal(et2, et)
    ctx.close()
