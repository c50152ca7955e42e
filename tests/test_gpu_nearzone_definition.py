"""The near-zone search's fast stages against its definition, the plain FP64
iteration, where the two could tell different results.  Scaling all lengths by
2^-100 scales every step of the plain iteration exactly and leaves FP32 no
squares to work with, so the scaled call takes the plain iteration for every
pair; the library's answer at scale 1 has to be the same, bit for bit."""
import numpy as np
import pytest

from synth import geometry as G
from tests._util import cuda

pytestmark = pytest.mark.gpu
Q = 10
CC = np.cos(np.pi * np.arange(Q + 1) / Q)


@pytest.fixture(scope="module")
def lib():
    from paper_1909_11085_gb300 import build
    build.build()
    import paper_1909_11085_gb300 as P
    return P


def _search(lib, nodes, npatch, x, d_eps, q=Q, scale=1.0):
    """(patch, uv, y, n, dist), lengths scaled back."""
    N, X = cuda(nodes * scale, x * scale)
    p, uv, y, n, d = (t.cpu().numpy() for t in
                      lib.near_patch_search(N, npatch, X, d_eps * scale, q))
    return p, uv, y / scale, n, np.where(p >= 0, d / scale, d)


def _wall_targets(rng, theta, z, R):
    rho = R - rng.uniform(0.05, 0.6, theta.size)
    return np.stack([rho * np.cos(theta), rho * np.sin(theta), z], 1)


@pytest.mark.parametrize("along", ["u", "v"])
def test_beside_a_node(lib, along):
    """A parameter 2e-9 to 8e-6 from a node, where the barycentric derivatives lose digits."""
    R, L, nth, nz = 6.0, 8.0, 6, 2
    nodes = G.cylinder_wall_patches(R, L, nth, nz, Q)[0]
    rng = np.random.default_rng(31)
    m = 300
    t = CC[rng.integers(1, Q, m)] + rng.choice([-1, 1], m) * np.exp(
        rng.uniform(np.log(2e-9), np.log(8e-6), m))
    o = 0.5 * (CC[3] + CC[4]) + 0.02 * rng.uniform(-1, 1, m)  # away from every node
    a, b = (t, o) if along == "u" else (o, t)
    theta = (rng.integers(0, nth, m) + 0.5 * (a + 1.0)) * 2 * np.pi / nth
    z = (rng.integers(0, nz, m) + 0.5 * (b + 1.0)) * L / nz
    x = _wall_targets(rng, theta, z, R)
    got, ref = (_search(lib, nodes, nth * nz, x, 1.0, scale=s) for s in (1.0, 2.0 ** -100))
    assert (ref[0] >= 0).all()
    for g, r in zip(got, ref):
        np.testing.assert_array_equal(g, r)
