"""The small direct form at the edges of its blocks (256 targets, tiles of 128
sources, 12 splits added at a time) and of its near-pair queue (none, some, more
than one batch, every pair of a tile), against the oracle."""
import numpy as np
import pytest

import oracle
from tests._util import cuda, max_rel, rel_l2

pytestmark = pytest.mark.gpu


@pytest.fixture(scope="module")
def lib():
    from paper_1909_11085_gb300 import build
    build.build()
    import paper_1909_11085_gb300 as P
    return P


# the bars of the mixed sums: 1e-6 in the 2-norm, 1e-5 in the maximum
@pytest.mark.parametrize("kind", ["sl", "dl", "sldl"])
@pytest.mark.parametrize("near", [0.0, 0.1, 10.0])  # h against coordinates in [-2, 2]
@pytest.mark.parametrize("ns,nt", [(1, 1), (2, 33), (127, 255), (129, 257), (1601, 70), (3001, 513)])
def test_sizes_and_near_shares(lib, kind, near, ns, nt):
    rng = np.random.default_rng(10 * ns + nt)
    src, trg = rng.uniform(-2, 2, (ns, 3)), rng.uniform(-2, 2, (nt, 3))
    trg[: min(ns, nt) // 3] = src[: min(ns, nt) // 3]  # coincident pairs contribute nothing
    f, phi, nrm = (rng.uniform(-1, 1, (ns, 3)) for _ in range(3))
    nrm /= np.linalg.norm(nrm, axis=1)[:, None]
    w, h = rng.uniform(0.5, 1.5, ns), np.full(ns, near)
    Y, F, N, PH, Wt, H, X = cuda(src, f, nrm, phi, w, h, trg)
    u0 = rng.uniform(-1e-3, 1e-3, (nt, 3))
    if kind == "sl":
        ref, call = oracle.sl(src, f, w, trg, 0.9), lambda **k: lib.sl(Y, F, Wt, X, 0.9, h=H, **k)
    elif kind == "dl":
        ref, call = oracle.dl(src, nrm, phi, w, trg), lambda **k: lib.dl(Y, N, PH, Wt, X, h=H, **k)
    else:
        ref = oracle.sldl(src, f, nrm, phi, w, trg, 0.9)
        call = lambda **k: lib.sldl(Y, F, N, PH, Wt, X, 0.9, h=H, **k)
    u = call(precision="mixed").cpu().numpy()
    assert rel_l2(u, ref) <= 1e-6, rel_l2(u, ref)
    assert max_rel(u, ref) <= 1e-5
    out, = cuda(u0)
    call(precision="mixed", out=out, accumulate=True)
    assert np.array_equal(out.cpu().numpy(), u0 + u)  # one FP64 sum: same rounding
