"""The FP64 far field with dense translations (kernel table and densities in fixed
point) over viscosities far from 1 and densities far from 1, against the host build of
the per-output passes.  The operators are random and scaled as the kernels are, so
that force and source densities carry velocities of one size at every viscosity."""
import numpy as np
import pytest

from synth import workloads as W
from tests import fmm_harness as H
from tests._util import cuda, rel_l2

pytestmark = pytest.mark.gpu
TOL = 1e-12  # the bar of the FP64 sums; the operators here do not amplify rounding


@pytest.fixture(scope="module")
def lib():
    from paper_1909_11085_gb300 import build
    build.build()
    from paper_1909_11085_gb300 import ops
    return ops


def _run(ops, kind, mu, size=1.0, p=4):
    wl = W.p2p_workload(ncell=6, radius=8.0, n_wall_patch=6, max_leaf=64)
    t = ops.octree(wl.pts, 64)
    o = t["perm"]
    t = ops.fmm_tree_arrays(**ops.fmm_tree_args(t))
    pts, f, phi, nrm, w = [a[o] for a in (wl.pts, wl.f, wl.phi, wl.nrm, wl.w)]
    flux = kind != "sl"
    ns, nc, D = p ** 3 - (p - 2) ** 3, 4 if flux else 3, t["max_depth"] - 1
    rng = np.random.default_rng(p)
    U = rng.uniform(-1, 1, (D, ns, nc, 3 * ns)) / ns
    U[:, :, :3] *= mu
    U = U.reshape(D, nc * ns, 3 * ns)
    V = mu * rng.uniform(-1, 1, (D, 3 * ns, 3 * ns)) / ns
    f = f * mu * size if kind != "dl" else None
    phi, nrm = (phi * size, nrm) if flux else (None, None)
    plan = ops.FmmFarPlan(t, p=p, mu=mu, flux=flux, uc2e=U, dc2e=V, m2l="dense", precision="fp64")
    got = plan(*cuda(pts, f, phi, nrm, w)).cpu().numpy()
    ref, _ = H.far_eval(pts, f, phi, nrm, w, t, p, U, V, mu, flux)
    s = np.abs(ref).max()
    assert s > 0
    return got / s, ref / s


@pytest.mark.parametrize("kind", ["sl", "dl", "sldl"])
@pytest.mark.parametrize("mu", [1e-18, 1e-9, 1e-3, 1.0, 1e6, 1e15])
def test_viscosities(lib, kind, mu):
    got, ref = _run(lib, kind, mu)
    assert rel_l2(got, ref) <= TOL


@pytest.mark.parametrize("size", [1e-305, 1e-100, 1e100])
def test_densities_of_any_size(lib, size):
    got, ref = _run(lib, "sldl", 1.0, size)
    assert rel_l2(got, ref) <= TOL
