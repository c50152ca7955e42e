"""The mixed far field at the lowest orders, whose CTAs have fewer threads than a batch has
source boxes, on a tree with V-lists of more than one batch, against the FP64 dense form
with the same operators."""
import numpy as np
import pytest

from synth import workloads as W
from tests._util import cuda, rel_l2
from tests.test_gpu_fmm import _oracle_ops

pytestmark = pytest.mark.gpu


@pytest.fixture(scope="module")
def lib():
    from paper_1909_11085_gb300 import build
    build.build()
    from paper_1909_11085_gb300 import ops
    return ops


# the mixed far field's bar, 1e-5
@pytest.mark.parametrize("p", [2, 3])
@pytest.mark.parametrize("m2l", ["dense", "fft"])
@pytest.mark.parametrize("flux", [False, True])
def test_low_orders(lib, p, m2l, flux):
    wl = W.p2p_workload(ncell=24, radius=8.0, n_wall_patch=6, max_leaf=16)
    t = lib.octree(wl.pts, 16)
    arrays = [a[t["perm"]] for a in (wl.pts, wl.f, wl.phi, wl.nrm, wl.w)]
    t = lib.fmm_tree_arrays(**lib.fmm_tree_args(t))
    assert np.diff(t["v_ptr"]).max() > 64
    by_depth = _oracle_ops(wl, t, p, flux)
    U = np.stack([by_depth[d][0] for d in sorted(by_depth)])
    D = np.stack([by_depth[d][1] for d in sorted(by_depth)])
    if not flux:
        arrays[2] = arrays[3] = None
    args = cuda(*arrays)
    plan, dense = (lib.FmmFarPlan(t, p=p, mu=wl.mu, flux=flux, uc2e=U, dc2e=D, m2l=m, precision=q)
                   for m, q in ((m2l, "mixed"), ("dense", "fp64")))
    got, ref = plan(*args).cpu().numpy(), dense(*args).cpu().numpy()
    assert rel_l2(got, ref) <= 1e-5, rel_l2(got, ref)
