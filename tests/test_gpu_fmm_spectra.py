"""The mixed far field with spectra, whose transforms and products take the parents
of all depths together and whose check-to-equivalent products take two or eight
boxes per CTA, on trees of few and many boxes per depth, against the FP64 dense
form with the same operators."""
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
@pytest.mark.parametrize("ncell,max_leaf", [(2, 64), (6, 300), (6, 8), (24, 8)])
@pytest.mark.parametrize("flux", [False, True])
def test_spectra_of_all_depths(lib, ncell, max_leaf, flux):
    wl = W.p2p_workload(ncell=ncell, radius=8.0, n_wall_patch=6, max_leaf=max_leaf)
    t = lib.octree(wl.pts, max_leaf)
    arrays = [a[t["perm"]] for a in (wl.pts, wl.f, wl.phi, wl.nrm, wl.w)]
    t = lib.fmm_tree_arrays(**lib.fmm_tree_args(t))
    assert t["max_depth"] >= 2
    by_depth = _oracle_ops(wl, t, 4, flux)
    U = np.stack([by_depth[d][0] for d in sorted(by_depth)])
    D = np.stack([by_depth[d][1] for d in sorted(by_depth)])
    if not flux:
        arrays[2] = arrays[3] = None
    args = cuda(*arrays)
    plan, dense = (lib.FmmFarPlan(t, p=4, mu=wl.mu, flux=flux, uc2e=U, dc2e=D, m2l=m, precision=q)
                   for m, q in (("fft", "mixed"), ("dense", "fp64")))
    got, ref = plan(*args).cpu().numpy(), dense(*args).cpu().numpy()
    assert rel_l2(got, ref) <= 1e-5, rel_l2(got, ref)
    assert np.array_equal(plan(*args).cpu().numpy(), got)
