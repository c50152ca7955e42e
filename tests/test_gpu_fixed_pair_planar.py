"""FP64 sums at the ends of the fixed point pair: double layers and gradients on a flat wall at targets from far to
very close above it, where every pair's difference is nearly perpendicular to the
normal: coordinates off the fixed point grid (a wall through the origin), on it
(a wall at z = 10) and a mixture, and densities below FP64's normal range, against the
oracle at the FP64 sums' bar."""
import numpy as np
import pytest

import oracle
from tests._util import cuda, rel_l2

pytestmark = pytest.mark.gpu
TOL64, GRAD64 = 1e-12, 1e-11


@pytest.fixture(scope="module")
def lib():
    from paper_1909_11085_gb300 import build
    build.build()
    import paper_1909_11085_gb300 as P
    return P


def _wall(rng, m, z0):
    a = (np.arange(m) + 0.5) / m * 60.0 - 30.0
    x, y = [v.ravel() for v in np.meshgrid(a, a, indexing="ij")]
    src = np.stack([x, y, np.full(m * m, z0)], 1)
    return src, np.tile([0.0, 0.0, 1.0], (m * m, 1)), rng.uniform(0.5, 1.5, m * m)


def _above(rng, nt, z0, h, few):
    z = z0 + h * rng.uniform(0.5, 1.0, nt)
    if few:  # one target in 20 that close, the others well above
        z = np.where(np.arange(nt) % 20 == 0, z, z0 + rng.uniform(2.0, 9.0, nt))
    return np.column_stack([rng.uniform(-28.0, 28.0, (nt, 2)), z])


@pytest.mark.parametrize("z0,few", [(0.0, False), (0.0, True), (10.0, False)])
@pytest.mark.parametrize("h", [1e-1, 1e-3, 1e-5, 1e-7, 1e-9, 1e-10])
def test_double_layer(lib, h, z0, few):
    rng = np.random.default_rng(41)
    src, nrm, w = _wall(rng, 40, z0)
    trg = _above(rng, 133, z0, h, few)
    near = slice(0, None, 20) if few else slice(None)
    for phi in (rng.uniform(-1, 1, src.shape), np.tile([0.0, 0.0, 1.0], (len(src), 1))):
        S, N, PH, Wt, T = cuda(src, nrm, phi, w, trg)
        got = lib.dl(S, N, PH, Wt, T, precision="fp64").cpu().numpy()
        ref = oracle.dl(src, nrm, phi, w, trg)
        assert rel_l2(got[near], ref[near]) <= TOL64
        assert rel_l2(got, ref) <= TOL64


@pytest.mark.parametrize("z0", [0.0, 10.0])
@pytest.mark.parametrize("h", [1e-2, 1e-6, 1e-9])
def test_gradients(lib, h, z0):
    rng = np.random.default_rng(42)
    src, nrm, w = _wall(rng, 20, z0)
    trg = _above(rng, 130, z0, h, False)
    phi = rng.uniform(-1, 1, src.shape)
    for g in (rng.uniform(-1, 1, trg.shape), np.tile([0.0, 0.0, 1.0], (len(trg), 1))):
        got = lib.sldl_grad(*[None if a is None else cuda(a)[0] for a in
                              (src, None, nrm, phi, w, trg, g)], 1.0, precision="fp64")
        ref = oracle.sldl_grad(src, None, nrm, phi, w, trg, g, 1.0)
        for k in ("phi", "y", "n", "x"):
            assert rel_l2(got[k].cpu().numpy(), ref["grad_" + k]) <= GRAD64


def test_subnormal_densities(lib):
    """Densities and velocities of some 1e-309, whose rounding of 5e-324 is far below the bar."""
    rng = np.random.default_rng(43)
    src, f = rng.uniform(-1, 1, (70, 3)), rng.uniform(-1, 1, (70, 3)) * 1e-309
    w = np.ones(70)
    S, F, Wt = cuda(src, f, w)
    got, ref = lib.sl(S, F, Wt, None, 1.0, precision="fp64").cpu().numpy(), oracle.sl(src, f, w, src)
    s = np.abs(ref).max()
    assert s > 0 and rel_l2(got / s, ref / s) <= TOL64
