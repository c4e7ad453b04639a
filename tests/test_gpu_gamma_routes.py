"""The Gamma form's kernels (linear up to 12 bins, rows up to 20, batches above) against the oracle's connection-
coefficient double sum and against each other: adding empty bins moves a context to the next kernel or
bin padding without changing the bins it had."""
import numpy as np
import pytest

from oracle import zeta_oracle as O

pytestmark = pytest.mark.gpu

torch = pytest.importorskip("torch")


def _fields(n, nb, seed):
    rng = np.random.Generator(np.random.PCG64(seed))
    return (rng.standard_normal((n, n, n)).astype(np.float32), rng.standard_normal((nb, n, n, n)).astype(np.float32))


@pytest.mark.parametrize("dsup", [2, 3, 4])
@pytest.mark.parametrize("nb", [1, 4, 7, 12, 13, 16, 20, 21])
def test_gamma_kernels(dsup, nb):
    from paper_2507_15209_gb300 import build
    build.build()
    from paper_2507_15209_gb300 import zeta as Z
    n = 16
    delta, a = _fields(n, nb, 10 * dsup + nb)
    ctx = Z.Context(n, 100.0, dsup, 0, np.linspace(5.0, 45.0, nb + 1), forms=("gamma",))
    d = torch.from_numpy(delta).cuda()
    got = ctx.sum_grid(d, Z.interleave(torch.from_numpy(a).cuda()), form="gamma").cpu().numpy()
    use = list(range(min(nb, 3)))  # the double sum of a few bins is enough of the oracle's time
    want = O.sum_gamma(delta.astype(np.float64), a[use].astype(np.float64), dsup)
    # 4096 cells (nodes) of up to 125 points in float32: random rounding of 6e-8 per product and tap
    scale = np.sqrt(np.abs(delta).astype(np.float64).mean() ** 2)
    assert np.abs(got[np.ix_(use, use)] - want).max() < 2e-6 * scale * 10
    np.testing.assert_array_equal(got, got.T)
    assert ctx.get_status() == 0
    ctx.close()


@pytest.mark.parametrize("dsup,n,most", [(2, 32, 12), (2, 32, 20), (3, 16, 20), (4, 32, 20)])
def test_rows_and_batches_agree(dsup, n, most):
    """The most bins of one kernel against the same bins and one empty (the next kernel or padding): the same
    products in another order of float32 sums, 1e-6 of the largest entry."""
    from paper_2507_15209_gb300 import zeta as Z
    delta, a = _fields(n, most, 77)
    d = torch.from_numpy(delta).cuda()
    out = []
    for nb in (most, most + 1):
        f = np.concatenate([a, np.zeros((nb - most, n, n, n), np.float32)])
        ctx = Z.Context(n, 100.0, dsup, 0, np.linspace(5.0, 45.0, nb + 1), forms=("gamma",))
        out.append(ctx.sum_grid(d, Z.interleave(torch.from_numpy(f).cuda()), form="gamma").cpu().numpy()[:most, :most])
        ctx.close()
    assert np.abs(out[0] - out[1]).max() < 1e-6 * max(np.abs(out[1]).max(), 1e-3)
