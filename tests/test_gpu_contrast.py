"""The contrast that the assignment writes, bit for bit against its float64 formula.

One particle on every node of a linear-basis grid (offset 0, so it lands whole on that node) makes the
fixed-point sum of a node its weight times a power of two, which the host forms exactly."""
import numpy as np
import pytest

pytestmark = pytest.mark.gpu

torch = pytest.importorskip("torch")


def _fma_less_one(v, inv):
    """float32(v inv - 1) with one float64 rounding: the product as an exact pair (Dekker), then a two-sum."""
    split = 134217729.0
    a = v * split
    vh = a - (a - v)
    b = inv * split
    ih = b - (b - inv)
    p = v * inv
    e = ((vh * ih - p) + vh * (inv - ih) + (v - vh) * ih) + (v - vh) * (inv - ih)
    s = p - 1.0
    bb = s - p
    return (s + (((p - (s - bb)) + (-1.0 - bb)) + e)).astype(np.float32)


@pytest.mark.parametrize("kind", ["ordinary", "near the mean", "signed", "sums"])
def test_contrast_bits(kind):
    from paper_2507_15209_gb300 import build
    build.build()
    from paper_2507_15209_gb300.zeta import Context, assign_noalloc
    n = 128
    rng = np.random.Generator(np.random.PCG64(11))
    k = np.arange(n, dtype=np.float32)
    z, y, x = np.meshgrid(k, k, k, indexing="ij")
    pos = np.stack([x, y, z], -1).reshape(-1, 3)
    m = len(pos)
    if kind == "ordinary":
        w = np.exp(rng.standard_normal(m)).astype(np.float32)
    elif kind == "near the mean":
        w = (1 + rng.integers(-64, 65, m) * 2.0 ** -23).astype(np.float32)
    else:
        w = (rng.standard_normal(m) + 0.3).astype(np.float32)
    # multiples of 2^-24, so that every weight is a whole number of the fixed-point units
    w = np.round(w.astype(np.float64) * 2.0 ** 24) / 2.0 ** 24
    w = w.astype(np.float32)
    node = np.arange(m)
    if kind == "sums":  # three weights on a node, far apart in size
        w2 = (np.round(np.exp(4 * rng.standard_normal(2 * m)) * 2.0 ** 16) / 2.0 ** 16).astype(np.float32)
        pos, w, node = np.concatenate([pos, pos, pos]), np.concatenate([w, w2]), np.concatenate([node, node, node])
    order = rng.permutation(len(w))
    parts = np.concatenate([pos, w[:, None]], 1)[order].astype(np.float32)
    dev = torch.from_numpy(parts).cuda()
    e = int(np.frexp(np.abs(w.astype(np.float64)).sum())[1])
    scale = 2.0 ** (61 - e)
    v = np.zeros(m, np.int64)
    np.add.at(v, node, np.rint(w.astype(np.float64) * scale).astype(np.int64))
    ctx = Context(n, float(n), 2, 0, np.array([3.0, 9.0]))
    delta, wsum = ctx.assign(dev)
    for d, s in ((delta, wsum), assign_noalloc(n, float(n), 2, dev)):
        inv = float(n) ** 3 / (float(s) * scale)
        np.testing.assert_array_equal(d.cpu().numpy().reshape(-1), _fma_less_one(v.astype(np.float64), inv))
    assert ctx.get_status() == 0
    ctx.close()
