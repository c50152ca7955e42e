"""Direct mixed sums whose source splits are cut into parts: whole FP32 summation
groups of 512 sources, ragged last group, near and coincident pairs in any part,
against the oracle and against the same 64 splits uncut."""
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


# The mixed bars (1e-6, 1e-5).  Cut and uncut add the same FP32 groups: into FP32
# (hi, lo) pairs, 2^-48 a step for at most 10 groups, and parts in FP64; 1e-12.
@pytest.mark.parametrize("kind", ["sl", "dl", "sldl"])
@pytest.mark.parametrize("ns,nt", [(140001, 1001), (300007, 225), (131072, 513)])
def test_parts(lib, kind, ns, nt):
    rng = np.random.default_rng(ns + nt)
    src, trg = rng.uniform(-2, 2, (ns, 3)), rng.uniform(-2, 2, (nt, 3))
    trg[::3] = src[:: ns // nt][: len(trg[::3])]
    f, phi, nrm = (rng.uniform(-1, 1, (ns, 3)) for _ in range(3))
    nrm /= np.linalg.norm(nrm, axis=1)[:, None]
    w, h = rng.uniform(0.5, 1.5, ns), np.full(ns, 0.15)
    Y, F, N, PH, Wt, H, X = cuda(src, f, nrm, phi, w, h, trg)
    if kind == "sl":
        ref = oracle.sl(src, f, w, trg, 0.9)
        call = lambda **k: lib.sl(Y, F, Wt, X, 0.9, h=H, **k)
    elif kind == "dl":
        ref = oracle.dl(src, nrm, phi, w, trg)
        call = lambda **k: lib.dl(Y, N, PH, Wt, X, h=H, **k)
    else:
        ref = oracle.sldl(src, f, nrm, phi, w, trg, 0.9)
        call = lambda **k: lib.sldl(Y, F, N, PH, Wt, X, 0.9, h=H, **k)
    u = call().cpu().numpy()
    assert rel_l2(u, ref) <= 1e-6, rel_l2(u, ref)
    assert max_rel(u, ref) <= 1e-5
    uncut = call(source_splits=64).cpu().numpy()
    assert rel_l2(u, uncut) <= 1e-12, rel_l2(u, uncut)
