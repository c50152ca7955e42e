"""FP64 gradients, whose pairs run in fixed point where they fit, at the ends of
that form: planar grids (zero differences and dots), pairs 1e-9 apart,
coordinates below the grid, a cloud far from the origin, one far outlier and
points out of the form's range (both take the plain FP64 pass), zero densities and
normals of very different lengths, against the oracle's analytic gradient."""
import numpy as np
import pytest

import oracle
from tests._util import cuda, rel_l2

pytestmark = pytest.mark.gpu
KEYS = {"f": "grad_f", "phi": "grad_phi", "y": "grad_y", "n": "grad_n", "x": "grad_x"}


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
    elif kind == "below":
        x[:: 20] *= 1e-7
        x[10:: 20] = x[:: 20][: len(x[10:: 20])] + 1e-4
    elif kind == "shifted":
        x += 1.0e6
    elif kind == "outlier":
        x *= 1e-3
        x[0] = 1e6
    elif kind == "large":
        x *= 2.0 ** 110  # past the exponents the fixed form takes
    return x


# the FP64 gradients' bar, 1e-11
@pytest.mark.parametrize("kind", ["sl", "dl", "sldl"])
@pytest.mark.parametrize("pts", ["uniform", "planar", "close", "below", "shifted", "outlier",
                                 "large"])
@pytest.mark.parametrize("ns,nt", [(1, 3), (37, 130), (300, 129)])
def test_grad_fp64(lib, kind, pts, ns, nt):
    rng = np.random.default_rng(11 * ns + nt)
    src = _points(pts, rng, ns)
    trg = np.concatenate([src[: nt // 2], _points(pts, rng, nt - min(nt // 2, ns))])
    f, phi, nrm = (rng.uniform(-1, 1, (ns, 3)) for _ in range(3))
    f[::3, 1] = 0.0
    phi[::5] = 0.0
    nrm[::7] = 0.0
    nrm[1::7] *= 1e-5
    g = rng.uniform(-1, 1, (nt, 3))
    w = rng.uniform(0.5, 1.5, ns)
    f = f if kind != "dl" else None
    phi, nrm = (phi, nrm) if kind != "sl" else (None, None)
    ref = oracle.sldl_grad(src, f, nrm, phi, w, trg, g, 0.9)
    Y, F, N, PH, Wt, X, G = cuda(src, f, nrm, phi, w, trg, g)
    out = lib.sldl_grad(Y, F, N, PH, Wt, X, G, 0.9, precision="fp64")
    for k, v in out.items():
        r, got = ref[KEYS[k]], v.cpu().numpy()
        assert np.isfinite(r).all()
        if np.abs(r).max() == 0.0:
            assert np.abs(got).max() == 0.0
        else:
            s = np.abs(r).max()
            assert rel_l2(got / s, r / s) <= 1e-11, (k, rel_l2(got / s, r / s))
