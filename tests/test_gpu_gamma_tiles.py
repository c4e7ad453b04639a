"""The Gamma form's kernels when a CTA walks several tiles, and every group of four bins against the oracle."""
import numpy as np
import pytest

from oracle import zeta_oracle as O

pytestmark = pytest.mark.gpu

torch = pytest.importorskip("torch")


def _fields(n, nb, seed):
    rng = np.random.Generator(np.random.PCG64(seed))
    return (rng.standard_normal((n, n, n)).astype(np.float32), rng.standard_normal((nb, n, n, n)).astype(np.float32))


def _size(Z, dsup):
    """A bound on the mean |term| of unit-variance fields: the B-spline filters average; the Daubechies ones are
    orthonormal, with weights whose signs differ."""
    return 1.0 if dsup != 3 else float(np.abs(Z.host_daub4_gamma()[1]).sum()) ** 3


@pytest.mark.parametrize("dsup", [2, 3, 4])
@pytest.mark.parametrize("nb", [12, 13, 16, 20, 21])
def test_several_tiles_per_cta(dsup, nb):
    """One CTA per SM takes three or four of the 512 tiles of a 64^3 grid, the default one.  The terms are the
    same; the float32 runs of at most 128 of them are cut elsewhere."""
    from paper_2507_15209_gb300 import build
    build.build()
    from paper_2507_15209_gb300 import zeta as Z
    n = 64
    delta, a = _fields(n, nb, 5 * dsup + nb)
    ctx = Z.Context(n, 100.0, dsup, 0, np.linspace(5.0, 45.0, nb + 1), forms=("gamma",))
    d, alm = torch.from_numpy(delta).cuda(), Z.interleave(torch.from_numpy(a).cuda())
    one = ctx.sum_grid(d, alm, form="gamma")
    tune = ctx.tuning()
    ctx.set_tuning([tune[0], tune[1], 1, *tune[3:]])
    many = ctx.sum_grid(d, alm, form="gamma")
    assert torch.cuda.get_device_properties(0).multi_processor_count < (n // 8) ** 3 // 2
    assert float((one - many).abs().max()) < 2 * 128 * 2.0 ** -24 * _size(Z, dsup)
    ctx.set_tuning(tune)
    assert torch.equal(ctx.sum_grid(d, alm, form="gamma"), one)
    assert ctx.get_status() == 0
    ctx.close()


@pytest.mark.parametrize("dsup", [2, 3, 4])
@pytest.mark.parametrize("nb", [10, 14, 20, 30])
def test_every_bin_group_against_oracle(dsup, nb):
    from paper_2507_15209_gb300 import zeta as Z
    n = 16
    delta, a = _fields(n, nb, 100 * dsup + nb)
    ctx = Z.Context(n, 100.0, dsup, 0, np.linspace(5.0, 45.0, nb + 1), forms=("gamma",))
    got = ctx.sum_grid(torch.from_numpy(delta).cuda(), Z.interleave(torch.from_numpy(a).cuda()), form="gamma").cpu().numpy()
    use = sorted({min(4 * g + g % 4, nb - 1) for g in range((nb + 3) // 4)} | {nb - 1})
    want = O.sum_gamma(delta.astype(np.float64), a[use].astype(np.float64), dsup)
    # a term is a product of values filtered three times with up to five taps (about 1e-6 of itself), and 4096
    # cells average those errors to 2e-8 of a term; the runs of 128 add less.  5e-7 of the largest mean |term|
    assert np.abs(got[np.ix_(use, use)] - want).max() < 5e-7 * _size(Z, dsup)
    assert ctx.get_status() == 0
    ctx.close()
