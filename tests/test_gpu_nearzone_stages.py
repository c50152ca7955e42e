"""The near-zone search's FP32 and FP64 stages against the brute-force oracle
over interpolation orders (the order whose loops are unrolled exactly and the
general ones), ragged target counts, coordinates far from the origin and
targets that only the plain FP64 iteration settles."""
import numpy as np
import pytest

from oracle import nearzone as NZ
from synth import geometry as G
from tests._util import cuda

pytestmark = pytest.mark.gpu


@pytest.fixture(scope="module")
def lib():
    from paper_1909_11085_gb300 import build
    build.build()
    import paper_1909_11085_gb300 as P
    return P


def _refined(nodes, npatch, q, x, d_eps):
    """The oracle's search, its point polished by Gauss-Newton steps inside the square:
    its minimiser stops where |x - P|^2 is flat to rounding, some 1e-8 from the minimum."""
    p, uv, y, n, d = NZ.near_patch_search(nodes, npatch, q, x, d_eps)
    X = np.asarray(nodes).reshape(npatch, -1, 3)
    for t in np.flatnonzero(p >= 0):
        z = uv[t].copy()
        for _ in range(60):
            P, Pu, Pv = [a[0] for a in NZ.patch_eval(X[p[t]], q, z[:1], z[1:])]
            J = np.stack([Pu, Pv], 1)
            g = J.T @ (P - x[t])
            free = ~(((z <= -1) & (g > 0)) | ((z >= 1) & (g < 0)))
            if not free.any():
                break
            step = np.zeros(2)
            step[free] = -np.linalg.solve((J.T @ J)[np.ix_(free, free)], g[free])
            z = np.clip(z + step, -1.0, 1.0)
        P, Pu, Pv = [a[0] for a in NZ.patch_eval(X[p[t]], q, z[:1], z[1:])]
        c = np.cross(Pu, Pv)
        y[t], n[t], d[t] = P, c / np.linalg.norm(c), np.linalg.norm(P - x[t])
    return p, y, n, d


def _check(lib, nodes, npatch, x, d_eps, q, scale=1.0):
    ref_p, ref_y, ref_n, ref_d = _refined(nodes, npatch, q, x, d_eps)
    N, X = cuda(nodes, x)
    p, uv, y, n, d = (t.cpu().numpy() for t in lib.near_patch_search(N, npatch, X, d_eps, q))
    hit = ref_p >= 0
    np.testing.assert_array_equal(p >= 0, hit)
    np.testing.assert_allclose(d[hit], ref_d[hit], rtol=0, atol=1e-9 * scale)
    np.testing.assert_allclose(y[hit], ref_y[hit], rtol=0, atol=1e-8 * scale)
    np.testing.assert_allclose(n[hit], ref_n[hit], rtol=0, atol=1e-7)
    # the parameters give the point: P(u, v) = y on the reported patch
    for i in np.flatnonzero(hit):
        P, _, _ = NZ.patch_eval(np.asarray(nodes).reshape(npatch, -1, 3)[p[i]], q, uv[i, :1],
                                uv[i, 1:])
        np.testing.assert_allclose(P[0], y[i], rtol=0, atol=1e-12 * max(1.0, np.abs(nodes).max()))
    assert (d[~hit] == -1).all() and (uv[~hit] == 0).all() and (y[~hit] == 0).all()


@pytest.mark.parametrize("q", [4, 6, 10, 12])
@pytest.mark.parametrize("m", [1, 33])
def test_orders(lib, q, m):
    cp = G.cubed_sphere_patches(1.2, q, 1)[0]
    rng = np.random.default_rng(100 * q + m)
    d = rng.normal(size=(m, 3))
    d /= np.linalg.norm(d, axis=1)[:, None]
    _check(lib, cp, 6, d * (1.2 + rng.uniform(-0.3, 0.4, m))[:, None], 0.25, q)


@pytest.mark.parametrize("shift", [0.0, 3.0e3])
def test_far_from_the_origin(lib, shift):
    cp = G.cylinder_wall_patches(6.0, 8.0, 6, 2, 10)[0] + shift
    rng = np.random.default_rng(21)
    th, rho = rng.uniform(0, 2 * np.pi, 24), 6.0 + rng.uniform(-1.5, 0.6, 24)
    x = np.stack([rho * np.cos(th), rho * np.sin(th), rng.uniform(0.5, 7.5, 24)], 1) + shift
    _check(lib, cp, 12, x, 1.0, 10, scale=10.0 if shift else 1.0)


def test_nodes_edges_and_repeats(lib):
    """Targets on nodes (distance exactly 0), a hair off them, past the ends of an
    open wall (closest points on an edge or a corner), each several times over,
    so that one cell holds many more targets than a warp."""
    q = 10
    cp = G.cylinder_wall_patches(6.0, 8.0, 6, 2, q)[0]
    rng = np.random.default_rng(22)
    on = cp[rng.choice(len(cp), 9, replace=False)]
    th = rng.uniform(0, 2 * np.pi, 8)
    past = np.stack([6.2 * np.cos(th), 6.2 * np.sin(th), np.where(th > 3.0, 8.4, -0.4)], 1)
    x = np.concatenate([on, on + 1e-9, on * (1.0 - 1e-13), past])
    _check(lib, cp, 12, x, 0.7, q)
    N, X = cuda(cp, np.tile(x, (9, 1)))
    got = [t.cpu().numpy() for t in lib.near_patch_search(N, 12, X, 0.7, q)]
    for a in got:  # every copy of a target has the same answer
        a = a.reshape(9, len(x), -1)
        assert (a == a[:1]).all()
    assert (got[4][:9] == 0.0).all()
