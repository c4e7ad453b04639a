"""The uniform term and the 2PCF from the per-|n|^2 sums against the FP64 oracle, over the range of the
half spectrum's size: ordinary contrasts, contrasts scaled by large and small powers, and a spectrum
that is only 8-byte aligned; non-finite spectra give non-finite results, a zero spectrum zero."""
import numpy as np
import pytest

from oracle import zeta_oracle as O
from paper_2507_15209_gb300 import mocks

pytestmark = pytest.mark.gpu

torch = pytest.importorskip("torch")


@pytest.mark.parametrize("n,dsup,scale", [(16, 2, 1.0), (32, 4, 1.0), (32, 3, 2.0 ** 40), (16, 4, 2.0 ** -40)])
def test_uniform_term_and_xi(n, dsup, scale):
    from paper_2507_15209_gb300 import build
    build.build()
    from paper_2507_15209_gb300.zeta import Context
    box, nb, lmax = 200.0, 5, 3
    edges = np.linspace(15.0, 80.0, nb + 1)
    delta = (mocks.lognormal_density(n, 9) - 1.0).astype(np.float32)
    ctx = Context(n, box, dsup, lmax, edges, forms=("node",))
    dhat = ctx.fft_r2c(torch.from_numpy(delta).cuda()) * scale
    # the same float32 spectrum in the oracle, Hermitian-completed; |delta_hat|^2 is all it uses
    d64 = dhat.double().cpu().numpy()
    half = np.zeros((n, n, n // 2 + 1), np.complex128)
    half[..., : n // 2] = d64[..., 0] + 1j * d64[..., 1]
    full = np.zeros((n, n, n), np.complex128)
    full[..., : n // 2 + 1] = half
    for x in range(1, n // 2):
        full[..., n - x] = np.conj(np.roll(half[::-1, ::-1, x], (1, 1), (0, 1)))
    odd = torch.empty(dhat.numel() + 2, device="cuda")[2:].view(dhat.shape)
    odd.copy_(dhat)
    assert odd.data_ptr() % 16 == 8
    for l in range(lmax + 1):
        got = ctx.mass_term(odd, l).cpu().numpy()
        want = O.mass_term_fourier(full, l, n, box, edges, dsup)
        # float32 window-table entries (6e-8 each, two per product) and float32 Gram chunks
        assert np.linalg.norm(got - want) < 1e-6 * np.linalg.norm(want)
    radii = np.array([0.0, 20.0, 55.5])
    xi = ctx.xi_radii(dhat, radii).cpu().numpy()
    iv = O.fft_integers(n)
    k = 2 * np.pi / box * np.sqrt((iv[:, None, None] ** 2 + iv[None, :, None] ** 2 + iv[None, None] ** 2).astype(float))
    p = np.abs(full) ** 2 * ~O.nyquist_mask(n)
    want = np.array([(p * np.sinc(k * r / np.pi)).sum() for r in radii]) / float(n) ** 6
    # exact to the pair arithmetic (2^-46) and the unit (2^-46 of the largest mode) of every mode
    assert np.abs(xi - want).max() < 1e-11 * want[0]
    assert ctx.get_status() == 0


def test_degenerate_spectra():
    from paper_2507_15209_gb300.zeta import Context
    n = 16
    ctx = Context(n, 100.0, 2, 1, np.array([10.0, 20.0, 30.0]), forms=("node",))
    dhat = torch.zeros((n, n, n // 2, 2), device="cuda")
    assert float(ctx.mass_term(dhat, 0).abs().max()) == 0
    for bad in (float("inf"), float("nan")):
        dhat[1, 2, 3, 0] = bad
        assert not torch.isfinite(ctx.mass_term(dhat, 1)).any()
    assert not torch.isfinite(ctx.xi_radii(dhat, [5.0])).any()
