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


def _strips(n, fold):
    """n square patches in a row along x, folded down by `fold` more at each shared edge (of
    constant u, with the same nodes on both sides), the last index first in space when odd."""
    out, at, ang = [], np.zeros(2), 0.0
    V = np.tile(CC, (Q + 1, 1))
    for _ in range(n):
        step = np.array([np.cos(ang), -np.sin(ang)])
        s = 1.0 - CC  # u = 1 at the start of the patch
        line = at + s[:, None] * step
        line[0] = at
        at = line[-1].copy()
        ang += fold
        out.append(np.stack([np.repeat(line[:, 0], Q + 1), V.ravel(),
                             np.repeat(line[:, 1], Q + 1)], 1))
    return np.stack(out)


@pytest.mark.parametrize("flip", [False, True])
def test_ties_on_an_edge(lib, flip):
    """Targets beyond a convex edge have their closest point on it: both patches hold it, and
    the lower index wins."""
    nodes = _strips(2, 0.9) + np.array([0.3, 0.7, -0.2])
    edge = nodes[0, -1]
    np.testing.assert_array_equal(nodes[0, -(Q + 1):], nodes[1, :Q + 1])
    nodes = (nodes[::-1] if flip else nodes).reshape(-1, 3)
    rng = np.random.default_rng(32)
    m = 600
    ang = rng.uniform(0.1, 0.8, m)  # between the two patches' normals
    out = np.stack([np.sin(ang), 0 * ang, np.cos(ang)], 1)
    x = np.stack([np.full(m, edge[0]), 0.7 + rng.uniform(-0.95, 0.95, m), np.full(m, edge[2])], 1)
    x = x + rng.uniform(0.01, 0.3, m)[:, None] * out
    p, uv, y, n, d = _search(lib, nodes, 2, x, 0.4)
    assert (p == 0).all()
    ref = _search(lib, nodes, 2, x, 0.4, scale=2.0 ** -100)
    for g, r in zip((p, uv, y, n, d), ref):
        np.testing.assert_array_equal(g, r)


def test_cube_edges_and_corners(lib):
    """A cube's faces, whose edges run in different directions in the parameters: the patch
    is the definition's, ties or not."""
    u, v = [a.ravel() for a in np.meshgrid(CC, CC, indexing="ij")]
    faces = []
    for ax in range(3):
        for sg in (1.0, -1.0):
            c = np.zeros((u.size, 3))
            c[:, ax], c[:, (ax + 1) % 3], c[:, (ax + 2) % 3] = sg, sg * u, v
            faces.append(5.0 * c)
    nodes = np.concatenate(faces)
    rng = np.random.default_rng(33)
    x = rng.uniform(-6.0, 6.0, (4000, 3))
    got, ref = (_search(lib, nodes, 6, x, 1.0, scale=s) for s in (1.0, 2.0 ** -100))
    np.testing.assert_array_equal(got[0], ref[0])
    beyond = (np.abs(x) > 5.0).sum(1) > 1  # closest to an edge or a corner
    assert (ref[0][beyond] >= 0).sum() > 200
    hit = ref[0] >= 0
    np.testing.assert_allclose(got[2][hit], ref[2][hit], rtol=0, atol=1e-9)
    np.testing.assert_allclose(got[4][hit], ref[4][hit], rtol=0, atol=1e-12)


def test_distance_of_exactly_d_eps(lib):
    """d_eps set to a target's own distance, as the definition has it: found."""
    R, L, nth, nz = 6.0, 8.0, 6, 2
    nodes = G.cylinder_wall_patches(R, L, nth, nz, Q)[0]
    rng = np.random.default_rng(34)
    x = _wall_targets(rng, rng.uniform(0, 2 * np.pi, 40), rng.uniform(0.5, 7.5, 40), R)
    d = _search(lib, nodes, nth * nz, x, 1.0, scale=2.0 ** -100)[4]
    for i in range(40):
        p, _, _, _, di = _search(lib, nodes, nth * nz, x[i:i + 1], d[i])
        assert p[0] >= 0 and di[0] == d[i]
        assert _search(lib, nodes, nth * nz, x[i:i + 1], np.nextafter(d[i], 0.0))[0][0] == -1


@pytest.mark.parametrize("power", [-140, 30, 70, 140])
def test_lengths_out_of_fp32s_range(lib, power):
    """Lengths whose squares, or which themselves, leave FP32's range."""
    R, L, nth, nz = 6.0, 8.0, 6, 2
    nodes = G.cylinder_wall_patches(R, L, nth, nz, Q)[0]
    rng = np.random.default_rng(35)
    x = np.concatenate([_wall_targets(rng, rng.uniform(0, 2 * np.pi, 100),
                                      rng.uniform(0.5, 7.5, 100), R), rng.uniform(-9, 9, (100, 3))])
    got, ref = (_search(lib, nodes, nth * nz, x, 0.7, scale=2.0 ** s) for s in (power, -100))
    assert (ref[0] >= 0).sum() > 90
    np.testing.assert_array_equal(got[0], ref[0])
    np.testing.assert_allclose(got[2], ref[2], rtol=0, atol=1e-9)
    np.testing.assert_allclose(got[4], ref[4], rtol=0, atol=1e-12)
