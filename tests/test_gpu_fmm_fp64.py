"""The blocked FP64 far field (fixed point evaluations, kernel table for the
dense M2L) against the host build of the per-output passes, with random
well-scaled operators on both sides, over surface orders with and without the
table, leaf sizes below and above a CTA's targets, density kinds, a V-list entry
the table does not hold and a viscosity out of fixed point's range."""
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


def _case(ops, max_leaf):
    wl = W.p2p_workload(ncell=6, radius=8.0, n_wall_patch=6, max_leaf=max_leaf)
    t = ops.octree(wl.pts, max_leaf)
    o = t["perm"]
    return ops.fmm_tree_arrays(**ops.fmm_tree_args(t)), [a[o] for a in (wl.pts, wl.f, wl.phi,
                                                                         wl.nrm, wl.w)]


def _run(ops, t, arrays, p, kind, mu, m2l="dense"):
    pts, f, phi, nrm, w = arrays
    flux = kind != "sl"
    ns, nc, D = p ** 3 - (p - 2) ** 3, 4 if flux else 3, t["max_depth"] - 1
    rng = np.random.default_rng(p)
    U = rng.uniform(-1, 1, (D, nc * ns, 3 * ns)) / ns
    V = rng.uniform(-1, 1, (D, 3 * ns, 3 * ns)) / ns
    f = f if kind != "dl" else None
    phi, nrm = (phi, nrm) if flux else (None, None)
    plan = ops.FmmFarPlan(t, p=p, mu=mu, flux=flux, uc2e=U, dc2e=V, m2l=m2l, precision="fp64")
    got = plan(*cuda(pts, f, phi, nrm, w)).cpu().numpy()
    spec = ops.fmm_m2l_spectra(p, mu, flux) if m2l == "fft" else None
    ref, _ = H.far_eval(pts, f, phi, nrm, w, t, p, U, V, mu, flux, spec=spec)
    return got, ref


@pytest.mark.parametrize("p", [2, 3, 5, 6, 7])
def test_orders(lib, p):
    t, a = _case(lib, 64)
    got, ref = _run(lib, t, a, p, "sldl", 0.8)
    assert rel_l2(got, ref) <= TOL


@pytest.mark.parametrize("max_leaf", [8, 300])
@pytest.mark.parametrize("kind,m2l", [("sl", "dense"), ("dl", "dense"), ("sldl", "fft")])
def test_leaves_and_kinds(lib, max_leaf, kind, m2l):
    t, a = _case(lib, max_leaf)
    assert t["max_depth"] >= 2
    got, ref = _run(lib, t, a, 4, kind, 1.3, m2l)
    assert rel_l2(got, ref) <= TOL


def test_entry_outside_the_table(lib):
    """A V-list entry of another depth is evaluated kernel by kernel."""
    t, a = _case(lib, 32)
    d = t["depth"]
    b = int(np.flatnonzero((d == 3) & (np.diff(t["v_ptr"]) > 2))[0])
    t["v_idx"] = t["v_idx"].copy()
    t["v_idx"][t["v_ptr"][b] + 1] = int(np.flatnonzero(d == 2)[-1])
    got, ref = _run(lib, t, a, 4, "sldl", 1.0)
    assert rel_l2(got, ref) <= TOL


def test_viscosity_out_of_range(lib):
    t, a = _case(lib, 64)
    got, ref = _run(lib, t, a, 4, "sl", 1e120)
    s = np.abs(ref).max()
    assert s > 0 and rel_l2(got / s, ref / s) <= TOL
