"""On small grids a measurement takes several (l, m) pairs per launch.  Its result has to be the bits of the
single-step calls made pair by pair, at batch sizes that divide the pairs and that do not, with more
bins than the register-blocked Gram takes, and with the tensor-core Grams (one pair at a time)."""
import numpy as np
import pytest

from paper_2507_15209_gb300 import mocks

pytestmark = pytest.mark.gpu

torch = pytest.importorskip("torch")


@pytest.mark.parametrize("n,nb,lmax,dsup,gram", [
    (16, 1, 0, 2, "fp32"), (16, 3, 4, 4, "fp32"), (32, 9, 5, 3, "fp32"), (64, 8, 4, 2, "fp32"), (64, 13, 2, 4, "fp32"),
    (64, 21, 1, 2, "fp32"), (32, 32, 2, 4, "fp32"), (32, 6, 3, 2, "bf16x3"), (128, 2, 2, 4, "fp32"), (32, 5, 3, 4, "tf32")])
def test_batched_pairs_equal_single_steps(n, nb, lmax, dsup, gram):
    from paper_2507_15209_gb300 import build
    build.build()
    from paper_2507_15209_gb300.zeta import Context
    box = 300.0
    edges = np.linspace(12.0, 100.0, nb + 1)
    parts = mocks.lognormal_catalogue(n, 4001, box, 3, 4)
    parts[:, 3] = np.random.default_rng(5).uniform(0.5, 1.5, len(parts)).astype(np.float32)
    dev = torch.from_numpy(parts).cuda()
    forms = ("node", "gamma", "particle") if n <= 32 else ("node", "particle")
    ctx = Context(n, box, dsup, lmax, edges, gram=gram, np_max=len(parts), forms=forms)
    got = ctx.zeta_ell(particles=dev, forms=forms)
    delta, wsum = ctx.assign(dev)
    dhat = ctx.fft_r2c(delta)
    srt, start = ctx.sort_particles(dev)
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
            assert torch.equal(got[f][l], want[f]), (f, l)
    # one rank's share of the pairs, in slots
    a = ctx.reduce_lm(sum(ctx.zeta_lm(r, 3, particles=dev, forms=forms) for r in range(3)), forms=forms)
    for f in forms:
        assert torch.equal(a[f], got[f]), f
    assert ctx.get_status() == 0
    ctx.close()
