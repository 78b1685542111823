"""A NaN in B with every eigenpair wanted: an error, and soon.

The implicit QR of a matrix of NaNs never deflates; it gives up after 40 n + 100 sweeps in all (under a second
at order 150), whatever the number of records that they are spread over.
"""
import time

import pytest

torch = pytest.importorskip("torch")
pytestmark = pytest.mark.gpu

DEV = "cuda:0"


@pytest.mark.parametrize("n_vir", [12, 40, 150])
def test_nan_is_refused_in_time(n_vir):
    from paper_2603_16575_gb300 import Context, osvmp2
    g = torch.Generator(device=DEV).manual_seed(1)
    B = torch.randn((2, n_vir, 64), dtype=torch.float64, device=DEV, generator=g)
    f = torch.diag(torch.tensor([-1.0, -0.5], dtype=torch.float64, device=DEV))
    e = torch.linspace(0.1, 5.0, n_vir, dtype=torch.float64, device=DEV)
    ctx = Context(0)
    ctx.build_osv(f, e, 0.0, B=B)                    # (loads the kernels)
    bad = B.clone()
    bad[1] = float("nan")
    torch.cuda.synchronize()
    t = time.perf_counter()
    with pytest.raises(osvmp2.OSVMP2Error) as err:
        ctx.build_osv(f, e, 0.0, B=bad)
    assert err.value.code == osvmp2.STATUS_CODES["E_NUMERIC"]
    assert time.perf_counter() - t < 4.0
    assert list(ctx.build_osv(f, e, 0.0, B=B)) == [n_vir, n_vir]
    ctx.close()
