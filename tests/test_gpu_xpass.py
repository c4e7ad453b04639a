"""The direct-store x-pass (grids of 256^3 and more) gives the bits of the staged one (shape 1), also for
groups with missing fields, for an output that is only 16-byte aligned, and in bfloat16."""
import numpy as np
import pytest

pytestmark = pytest.mark.gpu

torch = pytest.importorskip("torch")


@pytest.mark.parametrize("n,nb", [(256, 1), (256, 4), (256, 7), (512, 2), (512, 5)])
def test_direct_stores_equal_staged_stores(n, nb):
    from paper_2507_15209_gb300 import build
    build.build()
    from paper_2507_15209_gb300.zeta import Context
    ctx = Context(n, 500.0, 4, 3, np.linspace(8.0, 90.0, nb + 1), forms=("node",))
    g = torch.Generator(device="cuda").manual_seed(n + nb)
    dhat = ctx.fft_r2c(torch.randn((n, n, n), device="cuda", generator=g))
    direct = ctx.reconstruct_alm(dhat, 3, -2)
    groups = (nb + 3) // 4
    odd = torch.empty(groups * n ** 3 * 4 + 4, device="cuda")[4:].view(groups, n, n, n, 4)
    assert odd.data_ptr() % 32 == 16
    ctx.reconstruct_alm(dhat, 3, -2, out=odd)
    ctx.set_shapes([0, 0, 1])
    staged = ctx.reconstruct_alm(dhat, 3, -2)
    torch.cuda.synchronize()
    assert torch.equal(direct, staged) and torch.equal(odd, staged)
    assert float(direct.abs().max()) > 0
    if nb % 4:
        assert float(direct[-1][..., nb % 4:].abs().max()) == 0
    assert ctx.get_status() == 0
    ctx.close()


def test_direct_bfloat16_fields_equal_staged():
    from paper_2507_15209_gb300.zeta import Context
    n = 256
    ctx = Context(n, 500.0, 4, 1, np.linspace(8.0, 90.0, 6), gram="bf16_fields", forms=("node",))
    g = torch.Generator(device="cuda").manual_seed(3)
    delta = torch.randn((n, n, n), device="cuda", generator=g)
    a = ctx.zeta_ell(delta=delta, forms=("node",))["node"]
    ctx.set_shapes([0, 0, 1])
    b = ctx.zeta_ell(delta=delta, forms=("node",))["node"]
    assert torch.equal(a, b)
    ctx.close()
