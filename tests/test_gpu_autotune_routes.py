"""The autotuner times launches of as many (l, m) pairs as the measurement takes: with one pair, with pairs that
share launches, in a workspace that holds fewer, on the tensor-core Gram and above 20 bins.  With what it chose
a measurement is still the bits of its single steps, and with the settings put back those of before."""
import numpy as np
import pytest

from paper_2507_15209_gb300 import mocks

pytestmark = pytest.mark.gpu

torch = pytest.importorskip("torch")


@pytest.mark.parametrize("n,nb,lmax,dsup,gram,forms,keep", [
    (16, 2, 0, 2, "fp32", ("node", "gamma", "particle"), 1.0), (32, 4, 3, 3, "fp32", ("node", "gamma", "particle"), 1.0),
    (32, 4, 3, 4, "bf16x3", ("node", "particle"), 1.0), (64, 21, 1, 4, "fp32", ("node", "particle"), 1.0),
    (64, 8, 2, 2, "fp32", ("node", "particle"), 0.5)])
def test_autotuned_results(n, nb, lmax, dsup, gram, forms, keep):
    from paper_2507_15209_gb300 import build
    build.build()
    from paper_2507_15209_gb300 import zeta as Z
    box = 300.0
    p = torch.from_numpy(mocks.lognormal_catalogue(n, 6001, box, 3, 4)).cuda()
    ctx = Z.Context(n, box, dsup, lmax, np.linspace(12.0, 100.0, nb + 1), gram=gram, np_max=len(p), forms=forms)
    size = int(ctx.workspace.numel() * keep) // 256 * 256
    Z._check("zeta_set_workspace", Z.lib().zeta_set_workspace(ctx._h, ctx.workspace.data_ptr(), size))
    settings = ctx.tuning(), ctx.staging(), ctx.shapes()
    before = ctx.zeta_ell(particles=p, forms=forms)
    assert all(1 <= t <= 8 for t in ctx.autotune(p, forms=forms))
    tuned = ctx.zeta_ell(particles=p, forms=forms)
    delta, wsum = ctx.assign(p)
    dhat = ctx.fft_r2c(delta)
    srt, start = ctx.sort_particles(p)
    for l in range(lmax + 1):
        want = {f: torch.zeros((nb, nb), dtype=torch.float64, device="cuda") for f in forms}
        ctx.mass_term(dhat, l, -1.0, gram=want["particle"])
        for m in range(-l, l + 1):
            alm = ctx.reconstruct_alm(dhat, l, m)
            for f in forms:
                if f == "particle":
                    ctx.sum_particles(srt, start, wsum, alm, gram=want[f])
                else:
                    ctx.sum_grid(delta, alm, form=f, gram=want[f])
        for f in forms:
            assert torch.equal(tuned[f][l], want[f]), (f, l)
    ctx.set_tuning(settings[0])
    ctx.set_staging(settings[1])
    ctx.set_shapes(settings[2])
    after = ctx.zeta_ell(particles=p, forms=forms)
    for f in forms:
        assert torch.equal(after[f], before[f]), f
    assert ctx.get_status() == 0
    ctx.close()
