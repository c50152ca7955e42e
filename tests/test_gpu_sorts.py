"""The Morton order, bounding box and sorts behind the work items, through
calls whose result depends on them: a sum whose items are built from sorted
targets is the FP64 sum of the same points in any order, at sizes around the
one-launch sort's limit and the radix sort's blocks, with repeated and
collinear points."""
import numpy as np
import pytest

from tests._util import cuda, rel_l2

pytestmark = pytest.mark.gpu


@pytest.fixture(scope="module")
def lib():
    from paper_1909_11085_gb300 import build
    build.build()
    import paper_1909_11085_gb300 as P
    return P


@pytest.mark.parametrize("nt", [1, 2, 255, 2049, 8192, 8193, 20000, 70001])
@pytest.mark.parametrize("pts", ["random", "same", "line"])
def test_targets_of_any_order(lib, nt, pts):
    rng = np.random.default_rng(nt)
    src, f, w = rng.uniform(-1, 1, (40, 3)), rng.uniform(-1, 1, (40, 3)), np.full(40, 0.1)
    trg = rng.uniform(-3, 3, (nt, 3))
    if pts == "same":
        trg[:] = trg[0]
    elif pts == "line":
        trg[:, :2] = 0.25
    S, F, Wt, T = cuda(src, f, w, trg)
    ref = lib.sl(S, F, Wt, T, precision="fp64").cpu().numpy()
    # source_splits = 1 takes the sorted work items at every size
    got = lib.sl(S, F, Wt, T, precision="mixed", source_splits=1).cpu().numpy()
    assert rel_l2(got, ref) <= 1e-6
