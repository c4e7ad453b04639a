"""The unit of the per-|n|^2 sums comes from the modes that enter them: what lies on the excluded Nyquist planes
changes no bit of the uniform term or the 2PCF, and a spectrum at high |k| alone, where the tables are
smallest, is summed as finely as any other."""
import numpy as np
import pytest

pytestmark = pytest.mark.gpu

torch = pytest.importorskip("torch")


def _spectrum(n, seed):
    g = torch.Generator(device="cuda").manual_seed(seed)
    return torch.randn((n, n, n // 2, 2), device="cuda", generator=g)


@pytest.mark.parametrize("dsup,plane", [(2, 1e6), (3, 1e18), (4, float("inf"))])
def test_nyquist_planes_do_not_enter(dsup, plane):
    from paper_2507_15209_gb300 import build
    build.build()
    from paper_2507_15209_gb300.zeta import Context
    n = 32
    ctx = Context(n, 200.0, dsup, 2, np.linspace(15.0, 80.0, 6))
    radii = np.array([0.0, 20.0, 55.5])
    out = []
    for v in (0.0, plane):
        d = _spectrum(n, 5)
        d[n // 2] = v  # z, then y
        d[:, n // 2] = v
        out.append([ctx.mass_term(d, l) for l in range(3)] + [ctx.xi_radii(d, radii)])
    for a, b in zip(*out):
        assert torch.isfinite(a).all() and float(a.abs().max()) > 0
        assert torch.equal(a, b)
    assert ctx.get_status() == 0


@pytest.mark.parametrize("dsup", [2, 4])
@pytest.mark.parametrize("scale", [1.0, 2.0 ** 61, 2.0 ** 63, 2.0 ** -70])
def test_high_k_alone(dsup, scale):
    from paper_2507_15209_gb300.zeta import Context, lib
    n = 32
    ctx = Context(n, 200.0, dsup, 0, np.linspace(15.0, 80.0, 6), phi_hat=True)
    f = np.abs(np.fft.fftfreq(n, 1.0 / n))
    high = (f >= n // 2 - 2) & (f < n // 2)
    keep = torch.from_numpy(high[:, None, None] & high[None, :, None] & high[None, None, : n // 2]).cuda()
    d = _spectrum(n, 6) * keep[..., None] * scale
    got = float(ctx.xi_radii(d, np.array([0.0]))[0])
    ph = np.empty(n)
    assert lib().zeta_host_phi_hat(n, dsup, ph.ctypes.data) == 0
    ph = ph.astype(np.float32).astype(np.float64)
    p = (d.double().cpu().numpy() ** 2).sum(-1) * ph[:, None, None] * ph[None, :, None] * ph[None, None, : n // 2]
    want = 2 * p.sum() / float(n) ** 6
    # 32 modes, each within half a unit (2^-51 of the largest at most) and 2^-57 of itself; float64 sums of few terms
    assert abs(got - want) < 32 * 2.0 ** -51 * want
    assert ctx.get_status() == 0
