"""A workspace too small for the pairs that could share launches, down to the size for one (l, m) pair at a time:
every call runs in it, nothing is written past its end, and the results are the bits of a full one."""
import numpy as np
import pytest

from paper_2507_15209_gb300 import mocks

pytestmark = pytest.mark.gpu

torch = pytest.importorskip("torch")


def _one_pair_bytes(Z, n, box, dsup, edges, np_max, forms):
    """The size of the same context with a single pair (lmax = 0)."""
    ctx = Z.Context(n, box, dsup, 0, edges, np_max=np_max, forms=forms)
    size = ctx.workspace.numel()
    ctx.close()
    return size


def _set(Z, ctx, nbytes):
    """A workspace of nbytes with a guard behind it."""
    buf = torch.full((nbytes + 4096,), 91, dtype=torch.uint8, device="cuda")
    Z._check("zeta_set_workspace", Z.lib().zeta_set_workspace(ctx._h, buf.data_ptr(), nbytes))
    return buf


@pytest.mark.parametrize("n,nb,lmax,dsup,npart", [(16, 3, 4, 2, 1500), (32, 6, 4, 4, 5001), (64, 8, 3, 4, 20001),
                                                  (128, 2, 2, 2, 30000)])
def test_smaller_workspaces(n, nb, lmax, dsup, npart):
    from paper_2507_15209_gb300 import build
    build.build()
    from paper_2507_15209_gb300 import zeta as Z
    box, forms = 300.0, ("node", "gamma", "particle")
    edges = np.linspace(12.0, 100.0, nb + 1)
    dev = torch.from_numpy(mocks.lognormal_catalogue(n, npart, box, 3, 4)).cuda()
    rnd = torch.from_numpy(mocks.lognormal_catalogue(n, npart, box, 5, 6)).cuda()
    wts = mocks.loss_weights(lmax, nb, 7)
    ctx = Z.Context(n, box, dsup, lmax, edges, np_max=npart, forms=forms + ("backward", "ss"))
    full = ctx.workspace.numel()

    def calls():
        num, den = ctx.zeta_ell_ss(dev, rnd, forms=("node", "gamma"))
        out = [*ctx.zeta_ell(particles=dev, forms=forms).values(), *num.values(), *den.values()]
        out += [*ctx.xi(particles=dev, forms=("node", "particle")).values()]
        delta, _ = ctx.assign(dev)
        return out + [delta, ctx.reconstruct_alm(ctx.fft_r2c(delta), lmax, 0), ctx.backward_node(delta, wts)]

    want = calls()
    least = _one_pair_bytes(Z, n, box, dsup, edges, npart, forms + ("backward", "ss"))
    assert least < full
    for size in (least, (least + full) // 512 * 256):
        buf = _set(Z, ctx, size)
        for a, b in zip(calls(), want):
            assert torch.equal(a, b)
        assert bool((buf[size:] == 91).all())
    only = _one_pair_bytes(Z, n, box, dsup, edges, npart, ("particle",))
    buf = _set(Z, ctx, only - 256)
    with pytest.raises(Z.ZetaError) as e:
        ctx.zeta_ell(particles=dev, forms=("particle",))
    assert e.value.code == -6
    assert ctx.get_status() == 0
    ctx.close()


@pytest.mark.parametrize("parts", [1.0, 2.5])
def test_batch_in_a_small_workspace(parts):
    from paper_2507_15209_gb300 import zeta as Z
    n, box, lmax, nb = 64, 300.0, 3, 8
    edges = np.linspace(12.0, 100.0, nb + 1)
    cats = [mocks.lognormal_catalogue(n, 4000 + 777 * i, box, 20 + i, 40 + i) for i in range(5)]
    most = max(len(c) for c in cats)
    offs = np.concatenate([[0], np.cumsum([len(c) for c in cats])])
    dev = torch.from_numpy(np.concatenate(cats)).cuda()
    ctx = Z.Context(n, box, 4, lmax, edges, np_max=most, forms=("node", "particle"))
    want = ctx.batch(dev, offs, forms=("node", "particle"))
    torch.cuda.synchronize()
    size = int(parts * _one_pair_bytes(Z, n, box, 4, edges, most, ("node", "particle"))) // 256 * 256
    assert size < ctx.workspace.numel()
    buf = _set(Z, ctx, size)
    got = ctx.batch(dev, offs, forms=("node", "particle"))
    assert torch.equal(got, want)
    assert bool((buf[size:] == 91).all())
    assert ctx.get_status() == 0
    ctx.close()
