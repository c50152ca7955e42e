"""GPU parity of the FP64 direct sums, whose pairs run in fixed point where they
fit, on inputs at the ends of that form: planar grids (zero differences and
dots), pairs 1e-9 apart, coordinates that run below the grid, clouds far from
the origin or of extreme scale, one far outlier (the plain FP64 engine), zero
densities, at sizes around the items' target and column counts."""
import numpy as np
import pytest

import oracle
from tests._util import cuda, rel_l2

pytestmark = pytest.mark.gpu
TOL64 = 1e-12


@pytest.fixture(scope="module")
def lib():
    from paper_1909_11085_gb300 import build
    build.build()
    import paper_1909_11085_gb300 as P
    return P


def _points(kind, rng, n):
    x = rng.uniform(-3.0, 3.0, (n, 3))
    if kind == "planar":
        x = np.round(x)
        x[:, 2] = 1.25
    elif kind == "close":
        x[1::2] = x[: n // 2] + 1e-9 * rng.uniform(-1, 1, (n // 2, 3))
    elif kind == "below":  # coordinates near zero lose bits on the grid
        x[:: 20] *= 1e-7
        x[10:: 20] = x[:: 20][: len(x[10:: 20])] + 1e-4
    elif kind == "shifted":
        x += 1.0e6
    elif kind == "outlier":
        x *= 1e-3
        x[0] = 1e6
    return x


# Whole powers of two scale the sums exactly (single layer 1 / s, double layer
# 1 / s^2); the oracle, whose r^5 leaves FP64's range there, runs unscaled.
SCALE = {"huge": 2.0 ** 215, "tiny": 2.0 ** -190}


@pytest.mark.parametrize("pts", ["uniform", "planar", "close", "below", "shifted", "outlier",
                                 "huge", "tiny"])
@pytest.mark.parametrize("ns,nt", [(1, 1), (37, 19), (70, 16), (300, 133)])
def test_direct_fp64(lib, pts, ns, nt):
    rng = np.random.default_rng(7 * ns + nt)
    src = _points(pts, rng, ns)
    trg = np.concatenate([src[: nt // 2], _points(pts, rng, nt - nt // 2)])
    f, phi, nrm = (rng.uniform(-1, 1, (ns, 3)) for _ in range(3))
    f[::3, 1] = 0.0
    phi[::5] = 0.0
    nrm[::7] = 0.0
    w = rng.uniform(0.5, 1.5, ns)
    s = SCALE.get(pts, 1.0)
    S, T, F, PH, N, Wt = cuda(s * src, s * trg, f, phi, nrm, w)
    sl, dl = oracle.sl(src, f, w, trg, 0.7) / s, oracle.dl(src, nrm, phi, w, trg) / s / s
    for got, ref in [
            (lib.sl(S, F, Wt, T, 0.7, precision="fp64"), sl),
            (lib.dl(S, N, PH, Wt, T, precision="fp64"), dl),
            (lib.sldl(S, F, N, PH, Wt, T, 0.7, precision="fp64"),
             sl + dl if s != 1.0 else oracle.sldl(src, f, nrm, phi, w, trg, 0.7))]:
        got = got.cpu().numpy()
        assert np.isfinite(ref).all()
        if np.abs(ref).max() == 0.0:
            assert np.abs(got).max() == 0.0
        else:
            scale = np.abs(ref).max()  # in range for the norms at every scale of the points
            assert rel_l2(got / scale, ref / scale) <= TOL64


def test_infinite_and_nan_densities_pass_through(lib):
    """A density that is not finite makes every other target's velocity not finite."""
    rng = np.random.default_rng(3)
    src, f, w = rng.uniform(-1, 1, (60, 3)), rng.uniform(-1, 1, (60, 3)), np.ones(60)
    for v in (np.inf, np.nan):
        g = f.copy()
        g[7, 1] = v
        S, G, Wt = cuda(src, g, w)
        u = lib.sl(S, G, Wt, None, 1.0, precision="fp64").cpu().numpy()
        bad = ~np.isfinite(u).all(axis=1)
        assert bad[np.arange(60) != 7].all()
