"""The adjoint passes at the edges of their blocks (128 output points of a CTA in
two halves of 64, tiles of 128 inputs, splits and their parts), per kernel
kind and precision, against the oracle's analytic gradient."""
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


# the bars of the gradients: 1e-11 in FP64, 1e-5 mixed
@pytest.mark.parametrize("precision,tol", [("fp64", 1e-11), ("mixed", 1e-5)])
@pytest.mark.parametrize("kind", ["sl", "dl", "sldl"])
@pytest.mark.parametrize("ns,nt", [(1, 1), (64, 65), (129, 128), (300, 31), (70, 2500)])
def test_sizes_and_kinds(lib, precision, tol, kind, ns, nt):
    rng = np.random.default_rng(1000 * ns + nt)
    src, trg = rng.uniform(-2, 2, (ns, 3)), rng.uniform(-2, 2, (nt, 3))
    trg[: min(ns, nt) // 3] = src[: min(ns, nt) // 3]  # coincident pairs contribute nothing
    f, phi, nrm = (rng.uniform(-1, 1, (ns, 3)) for _ in range(3))
    nrm /= np.linalg.norm(nrm, axis=1)[:, None]
    g = rng.uniform(-1, 1, (nt, 3))
    w, h = rng.uniform(0.5, 1.5, ns), np.full(ns, 0.2)
    f = f if kind != "dl" else None
    phi, nrm = (phi, nrm) if kind != "sl" else (None, None)
    ref = oracle.sldl_grad(src, f, nrm, phi, w, trg, g, 0.9)
    Y, F, N, PH, Wt, H, X, G = cuda(src, f, nrm, phi, w, h, trg, g)
    out = lib.sldl_grad(Y, F, N, PH, Wt, X, G, 0.9, h=H, precision=precision)
    for k, v in out.items():
        r = ref[KEYS[k]]
        got = v.cpu().numpy()
        if np.abs(r).max() == 0.0:
            assert np.abs(got).max() == 0.0
        else:
            assert rel_l2(got, r) <= tol, (k, rel_l2(got, r))
