"""FP64 contractions by integer slices on the tensor cores, through the entry points that use them.

T_ii, S, F and K of random systems against plain FP64 torch at the sizes where the kernel's tiling can go
wrong: K around one k-block (32) and one scale chunk (256), rows around a TMA box (32, 64) and a tile (128,
64 columns), OSV counts up to the whole virtual space.  Tolerance: an FP64 dot product of length K is
within K 2^-53 sum |a b|, the sliced one within K 2^-60 of the rows' largest products plus K / 256
roundings; both together stay below 4 K 2^-53 max|a| max|b| K, far from any indexing mistake.
"""
import numpy as np
import pytest

torch = pytest.importorskip("torch")
pytestmark = pytest.mark.gpu

DEV = "cuda:0"
EPS = 2.0 ** -53


def _system(n_occ, n_vir, n_aux, seed, scale=1.0, spread=0.0):
    g = torch.Generator(device=DEV).manual_seed(seed)
    B = torch.randn((n_occ, n_vir, n_aux), dtype=torch.float64, device=DEV, generator=g) * scale
    if spread:      # rows over many orders of magnitude
        B *= torch.exp(-spread * torch.rand((n_occ, n_vir, 1), dtype=torch.float64, device=DEV, generator=g))
    e = 0.1 + 4.9 * torch.rand(n_vir, dtype=torch.float64, device=DEV, generator=g)
    f = 1e-2 * torch.ones((n_occ, n_occ), dtype=torch.float64, device=DEV)
    f.fill_diagonal_(0.0)
    f += torch.diag(-1.5 + 1.2 * torch.rand(n_occ, dtype=torch.float64, device=DEV, generator=g))
    return B, e, f


@pytest.mark.parametrize("n_vir,n_aux", [(1, 1), (7, 31), (31, 33), (33, 64), (64, 255), (65, 256), (127, 257),
                                         (129, 288), (160, 511), (163, 513)])
@pytest.mark.parametrize("spread", [0.0, 25.0])
def test_pair_blocks_match_plain_fp64(n_vir, n_aux, spread):
    from paper_2603_16575_gb300 import Context
    B, e, f = _system(2, n_vir, n_aux, 100 + n_vir, spread=spread)
    ctx = Context(0)
    l_osv = 0.0 if n_vir < 100 else 1e-3       # the whole virtual space, and a truncated one
    k = ctx.build_osv(f, e, l_osv, B=B)
    Q = [ctx.get_osv(i)[0] for i in range(2)]
    for i in range(2):                         # T_ii through its eigenvalues
        T = (B[i] @ B[i].T) / (e[:, None] + e[None, :] - 2.0 * f[i, i])
        w = torch.linalg.eigvalsh(T).flip(0)[: int(k[i])]
        assert (ctx.get_osv(i)[1] - w).abs().max() <= 1e-12 * w[0]
    ctx.pair_integrals([(0, 1)], "fp64")
    P = torch.cat(Q, 1)
    K, S, F = ctx.get_pair_blocks(0, 1)
    G = [P.T @ B[i] for i in range(2)]
    size = float(P.abs().max()) * n_vir * float(B.abs().max())      # bound of |P^T B|
    tol_k = 4 * EPS * (n_aux * float(G[0].abs().max()) * float(G[1].abs().max()) * n_aux ** 0.5
                       + n_vir * size * float(max(x.abs().max() for x in G)) * n_aux)
    assert (K - G[0] @ G[1].T).abs().max() <= tol_k
    assert (S - P.T @ P).abs().max() <= 4 * EPS * n_vir
    assert (F - P.T @ (e[:, None] * P)).abs().max() <= 4 * EPS * n_vir * float(e.max())
    K0, S0, F0 = ctx.get_pair_blocks(0, 0)
    assert (S0 - Q[0].T @ Q[0]).abs().max() <= 4 * EPS * n_vir
    assert torch.equal(S0, S[: k[0], : k[0]])
    ctx.close()


@pytest.mark.parametrize("scale", [1e-100, 1e-30, 1e30])
def test_values_far_from_one(scale):
    """Exponents of the slices and of their sums outside FP32's range."""
    from paper_2603_16575_gb300 import Context
    B, e, f = _system(2, 40, 300, 3)
    ctx = Context(0)
    ctx.build_osv(f, e, 0.0, B=B)
    Q = [ctx.get_osv(i)[0] for i in range(2)]
    ctx.pair_integrals([(0, 1)], "fp64")
    K1 = ctx.get_pair_blocks(0, 1)[0]
    Bs = B * scale
    ctx.build_osv(f, e, 0.0, B=Bs)
    Qs = [ctx.get_osv(i)[0] for i in range(2)]
    ctx.pair_integrals([(0, 1)], "fp64")
    K2 = ctx.get_pair_blocks(0, 1)[0]
    P, Ps = torch.cat(Q, 1), torch.cat(Qs, 1)
    ref = (Ps.T @ B[0]) @ (Ps.T @ B[1]).T
    assert (K1 - (P.T @ B[0]) @ (P.T @ B[1]).T).abs().max() <= 1e-11 * ref.abs().max()
    assert (K2 / scale / scale - ref).abs().max() <= 1e-11 * ref.abs().max()
    ctx.close()
