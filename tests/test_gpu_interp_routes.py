"""The staged interpolation's halo copies (box copies inside, node copies at the faces) against the FP64
oracle and against the unstaged kernel, over grids with no, few and many inner tiles."""
import numpy as np
import pytest

from oracle import zeta_oracle as O

pytestmark = pytest.mark.gpu

torch = pytest.importorskip("torch")


@pytest.mark.parametrize("n,nb,dsup,npart", [(16, 3, 4, 700), (32, 5, 4, 9000), (32, 20, 4, 3000), (32, 27, 3, 3000),
                                             (64, 8, 4, 40000), (64, 6, 2, 40000)])
def test_staged_and_unstaged_sums(n, nb, dsup, npart):
    from paper_2507_15209_gb300 import build
    build.build()
    from paper_2507_15209_gb300 import zeta as Z
    box = 100.0
    rng = np.random.Generator(np.random.PCG64(n + nb))
    p = np.empty((npart, 4), np.float32)
    p[:, :3] = rng.random((npart, 3)) * box
    p[: npart // 3, :3] = (rng.random((npart // 3, 3)) * 6 + 10) * box / n  # a crowded corner: several batches a tile
    p[:, 3] = rng.random(npart) + 0.5
    p[p >= box] = 0.0
    a = rng.standard_normal((nb, n, n, n)).astype(np.float32)
    ctx = Z.Context(n, box, dsup, 0, np.linspace(2.0, 45.0, nb + 1), np_max=npart, forms=("particle",))
    srt, start = ctx.sort_particles(torch.from_numpy(p).cuda())
    w = torch.tensor([p[:, 3].astype(np.float64).sum()], device="cuda")
    alm = Z.interleave(torch.from_numpy(a).cuda())
    staged = ctx.sum_particles(srt, start, w, alm).cpu().numpy()
    ctx.set_staging(129)
    direct = ctx.sum_particles(srt, start, w, alm).cpu().numpy()
    want = O.sum_particles(a.astype(np.float64), p[:, :3].astype(np.float64), p[:, 3], n, box, dsup)
    # values of up to 64 float32 products (3e-7 of their size at worst), random over the particles
    size = np.sqrt(np.outer(np.diag(want), np.diag(want)))
    assert (np.abs(staged - want) < 3e-7 * size).all()
    assert (np.abs(direct - want) < 3e-7 * size).all()
    assert ctx.get_status() == 0
