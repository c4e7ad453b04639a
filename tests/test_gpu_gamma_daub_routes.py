"""The Gamma form of the Daubechies basis at 17 to 20 bins takes the row-ring kernel while a launch has no more
CTAs than SMs, and the batched kernel above.  A measurement whose pairs share a launch (batched) has to be the
bits of the single steps (rows), for the bins on both sides of the rule and for the cubic basis."""
import numpy as np
import pytest

from paper_2507_15209_gb300 import mocks

pytestmark = pytest.mark.gpu

torch = pytest.importorskip("torch")


@pytest.mark.parametrize("dsup,nb", [(3, 16), (3, 17), (3, 20), (4, 20)])
def test_shared_launches_equal_single_steps(dsup, nb):
    from paper_2507_15209_gb300 import build
    build.build()
    from paper_2507_15209_gb300.zeta import Context
    n, box, lmax = 32, 300.0, 2
    ctx = Context(n, box, dsup, lmax, np.linspace(12.0, 100.0, nb + 1), forms=("gamma",))
    delta = torch.from_numpy((mocks.lognormal_density(n, 3) - 1.0).astype(np.float32)).cuda()
    got = ctx.zeta_ell(delta=delta, forms=("gamma",))["gamma"]
    dhat = ctx.fft_r2c(delta)
    for l in range(lmax + 1):
        want = torch.zeros((nb, nb), dtype=torch.float64, device="cuda")
        for m in range(-l, l + 1):
            ctx.sum_grid(delta, ctx.reconstruct_alm(dhat, l, m), form="gamma", gram=want)
        assert float(want.abs().max()) > 0
        assert torch.equal(got[l], want), l
    assert ctx.get_status() == 0
    ctx.close()
