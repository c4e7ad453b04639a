"""Gradients at the bin counts, bases and grid sides where the adjoint kernels change form (bins padded to
fours, two- and four-node stencils, the 256^3 x-pass), against the oracle or the same call's linearity."""
import numpy as np
import pytest

from oracle import zeta_oracle as O
from paper_2507_15209_gb300 import mocks

pytestmark = pytest.mark.gpu

torch = pytest.importorskip("torch")


def _ctx(*a, **k):
    from paper_2507_15209_gb300 import build
    build.build()
    from paper_2507_15209_gb300.zeta import Context
    return Context(*a, **k)


# float32 gradients against float64: the bounds of the suite's other gradient tests (2e-5 node, 1e-4 particle)
@pytest.mark.parametrize("nb", [1, 5, 13, 18, 32])
@pytest.mark.parametrize("dsup", [2, 4])
def test_gradients_against_oracle(nb, dsup):
    n, box, lmax = 16, 90.0, 2
    edges = np.linspace(7.0, 40.0, nb + 1)
    parts = mocks.lognormal_catalogue(n, 1203, box, 31, 32)
    parts[:, 3] = np.random.default_rng(33).uniform(0.5, 1.5, len(parts)).astype(np.float32)
    wts = mocks.loss_weights(lmax, nb, 34)
    ctx = _ctx(n, box, dsup, lmax, edges, np_max=len(parts), forms=("particle", "backward"))
    got = ctx.backward_particles(torch.from_numpy(parts).cuda(), wts).cpu().numpy()
    want = O.grad_particle_positions(parts.astype(np.float64), wts, n, box, edges, lmax, dsup)
    assert np.linalg.norm(got - want) < 1e-4 * np.linalg.norm(want)
    delta = (mocks.lognormal_density(n, 35) - 1.0).astype(np.float32)
    got = ctx.backward_node(torch.from_numpy(delta).cuda(), wts).cpu().numpy()
    want = O.grad_node_delta(delta.astype(np.float64), wts, n, box, edges, lmax)
    assert np.linalg.norm(got - want) < 2e-5 * np.linalg.norm(want)
    assert ctx.get_status() == 0


@pytest.mark.parametrize("n,nb", [(256, 5), (512, 2)])
def test_node_gradient_by_euler_identity(n, nb):
    """zeta_node is a cubic form of delta, so delta . dL/d delta = 3 L, on the grids whose x-pass has its own
    kernel.  Both sides are sums over n^3 float32 products: 2e-5 of their size."""
    lmax = 1
    edges = np.linspace(10.0, 80.0, nb + 1)
    wts = mocks.loss_weights(lmax, nb, 41)
    ctx = _ctx(n, 500.0, 4, lmax, edges, forms=("node", "backward"))
    g = torch.Generator(device="cuda").manual_seed(5)
    delta = torch.exp(torch.randn((n, n, n), device="cuda", generator=g)) - 1.6
    z = ctx.zeta_ell(delta=delta, forms=("node",))["node"]
    w = torch.from_numpy(wts).cuda()
    size = float((w.abs() * z.abs()).sum())
    grad = ctx.backward_node(delta, wts)
    assert abs(float((grad.double() * delta.double()).sum()) - 3 * float((w * z).sum())) < 3 * 2e-5 * size
    assert ctx.get_status() == 0
