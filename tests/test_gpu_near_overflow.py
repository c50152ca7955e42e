"""The U-list near field where candidate lists overflow: few, some and nearly all of its
items, below and above the number of items from which on a warp takes
each instead of a CTA, in all kinds, against the oracle at sampled targets."""
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


# Leaves of 25.6 points on average, 27 of them in an inner leaf's U-list: 691 sources, of which
# one leaf edge about the leaf's box holds some 528, two edges all; a list holds 512.
@pytest.fixture(scope="module", params=[4, 5])
def case(request, lib):
    depth = request.param
    rng = np.random.default_rng(51)
    n = int(25.6 * 8 ** depth / 4)
    pts = rng.uniform(-1, 1, (n, 3)) * [1.0, 0.5, 0.5]
    pts[:2] = [[-1.0, -0.5, -0.5], [1.0, 0.5, 0.5]]
    t = lib.octree(pts, 64)
    pts = pts[t["perm"]]
    f, phi, nrm = (rng.uniform(-1, 1, (n, 3)) for _ in range(3))
    nrm /= np.linalg.norm(nrm, axis=1)[:, None]
    w, h = rng.uniform(0.5, 1.5, n), np.full(n, 2.0 / 2 ** depth / 3.0)
    nleaf = len(t["leaf_ptr"]) - 1
    assert nleaf > (4864 if depth == 5 else 500)
    pick = np.asarray(t["leaf_ptr"])[np.linspace(0, nleaf - 1, 60).astype(int)]
    return t, pts, f, phi, nrm, w, h, np.unique(pick)


@pytest.mark.parametrize("kernels", [1, 2, 3])
@pytest.mark.parametrize("near_ratio", [0.5, 3.0, 6.0])
def test_parity(lib, case, near_ratio, kernels):
    t, pts, f, phi, nrm, w, h, pick = case
    plan = lib.P2PPlan(len(pts), t["leaf_ptr"], t["ulist_ptr"], t["ulist_idx"], kernels, "mixed",
                       near_ratio)
    X, F, P, N, W, H = cuda(pts, f, phi, nrm, w, h)
    got = [plan(X, f=F if kernels & 1 else None, phi=P if kernels & 2 else None,
                nrm=N if kernels & 2 else None, w=W, h=H).cpu().numpy()[pick] for _ in range(2)]
    plan.device_status()
    np.testing.assert_array_equal(got[0], got[1])  # whichever warp took an item
    ref = oracle.p2p(pts, f, phi, nrm, w, t["leaf_ptr"], t["ulist_ptr"], t["ulist_idx"], kernels,
                     1.0, targets=pick)
    assert rel_l2(got[0], ref) <= 1e-6
    assert max_rel(got[0], ref) <= 1e-5


def test_replayed_from_a_graph(lib, case):
    t, pts, f, phi, nrm, w, h, pick = case
    plan = lib.P2PPlan(len(pts), t["leaf_ptr"], t["ulist_ptr"], t["ulist_idx"], 3, "mixed", 6.0)
    args = cuda(pts, f, phi, nrm, w)
    H = cuda(h)[0]
    ref = plan(*args, h=H).cpu().numpy()
    graph = plan.capture(*args, h=H)
    for _ in range(2):
        np.testing.assert_array_equal(graph.launch().cpu().numpy(), ref)
