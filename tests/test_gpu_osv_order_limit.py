"""Virtual spaces beyond the exact eigen-solver's shared memory are refused before anything is launched: from order
9537 on no warp's staging rows are left beside the vectors of a step, and nothing of the matrix would be swept."""
import pytest

torch = pytest.importorskip("torch")
pytestmark = pytest.mark.gpu

DEV = "cuda:0"


@pytest.mark.parametrize("n_vir", [9537, 9632, 9633, 12000])
@pytest.mark.parametrize("l_osv,prec", [(1e-4, "fp64"), (1e-4, "mixed"), (0.0, "fp64")])
def test_orders_beyond_the_limit_are_refused(n_vir, l_osv, prec):
    from paper_2603_16575_gb300 import Context, osvmp2
    ctx = Context(0, osv_prec=prec)
    f = torch.tensor([[-1.0]], dtype=torch.float64, device=DEV)
    e = torch.linspace(0.1, 5.0, n_vir, dtype=torch.float64, device=DEV)
    env = torch.full((1, n_vir), 0.1, dtype=torch.float64, device=DEV)
    torch.cuda.synchronize()
    before = osvmp2.kernel_launches()
    with pytest.raises(osvmp2.OSVMP2Error) as err:
        ctx.build_osv(f, e, l_osv, env=env, seed=1, n_aux=8)
    assert err.value.code == osvmp2.STATUS_CODES["E_ARG"]
    assert osvmp2.kernel_launches() == before
    # the context is usable
    assert ctx.build_osv(f, e[:40].contiguous(), 1e-6, env=env[:, :40].contiguous(), seed=1, n_aux=8)[0] > 0
    ctx.close()
