"""The routes of the assignment (direct scatter, records grouped by tile, prepared sorted records) against
the FP64 oracle, with particles at cell faces, at the box edge and outside the box."""
import numpy as np
import pytest

from oracle import zeta_oracle as O

pytestmark = pytest.mark.gpu

torch = pytest.importorskip("torch")


def _particles(n, box, npart, seed):
    rng = np.random.Generator(np.random.PCG64(seed))
    p = np.empty((npart, 4), np.float32)
    p[:, :3] = rng.random((npart, 3)) * box
    faces = rng.integers(0, n + 1, (npart // 8, 3)) * (box / n)
    p[: npart // 8, :3] = faces
    p[npart // 8 : npart // 4, 0] = np.nextafter(p[npart // 8 : npart // 4, 0], np.float32(0))
    p[0, :3] = (0.0, np.nextafter(np.float32(box), np.float32(0)), box)
    p[1, :3] = (-1e-3, 1e-7, box * 1.25)
    p[:, 3] = rng.random(npart) + 0.5
    p[2, 3] = 0.0
    p[3, 3] = -0.25
    return p


# (n, D, particles): 256^3 with at least 2^24 / 64 particles groups the records, one fewer does not
@pytest.mark.parametrize("n,dsup,npart", [(16, 2, 1), (16, 4, 33), (64, 3, 5001), (128, 4, 3000), (256, 4, 262143),
                                          (256, 4, 262144), (256, 3, 262145)])
def test_assign_routes_against_oracle(n, dsup, npart):
    from paper_2507_15209_gb300 import build
    build.build()
    from paper_2507_15209_gb300.zeta import Context
    box = 1000.0
    p = _particles(n, box, max(npart, 4), 7)[:npart]
    if npart == 1:
        p[0, 3] = 1.0
    dev = torch.from_numpy(p).to("cuda")
    ctx = Context(n, box, dsup, 0, np.array([10.0, 60.0]), np_max=npart, forms=("particle",))
    delta, wsum = ctx.assign(dev)
    eps, w = O.assign(p[:, :3].astype(np.float64), p[:, 3].astype(np.float64), n, box, dsup)
    want = O.contrast(eps, w)
    # float32 weights: each factor within 6e-7 of itself (or 1e-7 of the largest), the product of three
    # within 2e-6; a contribution is at most n^3 / W of the contrast, and at most `most` of them meet
    cell = np.floor(p[:, :3].astype(np.float64) * (n / box)).astype(np.int64) % n
    most = np.unique(cell, axis=0, return_counts=True)[1].max()
    tol = 3e-6 * (1 + np.abs(want)) + 3e-7 * most * n ** 3 / abs(w)
    assert abs(float(wsum) - w) <= 1e-12 * np.abs(p[:, 3]).sum()
    assert np.all(np.abs(delta.cpu().numpy() - want) <= tol)
    # the sorted route inside a measurement: the same fixed-point sums, so the same grid
    a = ctx.zeta_ell(particles=dev, forms=("particle",))["particle"]
    b = ctx.zeta_ell(particles=dev, delta=delta, forms=("particle",))["particle"]
    torch.cuda.synchronize()
    assert torch.equal(a, b)
    assert ctx.get_status() == 0
