"""More kept OSVs than a CTA's warps take in one round of inverse iteration, in a large virtual space: one CTA per matrix
(more orbitals than clusters of two fit the GPU), order above 16 x 176, more than 512 vectors kept.

Tolerances as for the smaller orders: a few n eps ||T||_F for eigenvalues and residuals, a few n eps for the overlaps.
"""
import pytest

torch = pytest.importorskip("torch")
pytestmark = pytest.mark.gpu

DEV = "cuda:0"
EPS = 2.0 ** -53


def test_kept_vectors_beyond_one_round_of_inverse_iteration():
    from paper_2603_16575_gb300 import Context
    n_occ, n_vir, n_aux = 150, 3008, 600
    g = torch.Generator(device=DEV).manual_seed(5)
    env = 0.05 + 0.05 * torch.rand((n_occ, n_vir), dtype=torch.float64, device=DEV, generator=g)
    e = 0.1 + 4.9 * torch.rand(n_vir, dtype=torch.float64, device=DEV, generator=g)
    f = torch.diag(-1.5 + 1.2 * torch.rand(n_occ, dtype=torch.float64, device=DEV, generator=g))
    from paper_2603_16575_gb300 import osvmp2
    ctx = Context(0)
    k = ctx.build_osv(f, e, 1e-3, env=env, seed=3, n_aux=n_aux)
    assert min(k) > 16 * 32
    for i in (0, 71, 149):
        B = osvmp2.generate_B(n_occ, n_vir, n_aux, 3, env, i0=i, n_i=1)[0]
        T = (B @ B.T) / (e[:, None] + e[None, :] - 2.0 * f[i, i])
        Q, w = ctx.get_osv(i)
        frob = float(torch.linalg.norm(T))
        assert (T @ Q - Q * w).abs().max() <= 8 * n_vir * EPS * frob
        assert (Q.T @ Q - torch.eye(Q.shape[1], dtype=Q.dtype, device=DEV)).abs().max() <= 8 * n_vir * EPS
    ctx.close()
