"""FP64 far-field plans of different orders called from two host threads at once:
every call succeeds and gives the plan's own result."""
import threading

import numpy as np
import pytest

from synth import workloads as W
from tests._util import cuda

pytestmark = pytest.mark.gpu


@pytest.fixture(scope="module")
def lib():
    from paper_1909_11085_gb300 import build
    build.build()
    from paper_1909_11085_gb300 import ops
    return ops


def test_orders_on_two_threads(lib):
    import torch

    wl = W.p2p_workload(ncell=6, radius=8.0, n_wall_patch=6, max_leaf=64)
    t = lib.octree(wl.pts, 64)
    o = t["perm"]
    t = lib.fmm_tree_arrays(**lib.fmm_tree_args(t))
    arrays = cuda(*[a[o] for a in (wl.pts, wl.f, wl.phi, wl.nrm, wl.w)])
    plans, ref = [], []
    for p in (2, 6):
        ns, D = p ** 3 - (p - 2) ** 3, t["max_depth"] - 1
        rng = np.random.default_rng(p)
        plans.append(lib.FmmFarPlan(t, p=p, mu=1.0, flux=True, m2l="dense", precision="fp64",
                                    uc2e=rng.uniform(-1, 1, (D, 4 * ns, 3 * ns)) / ns,
                                    dc2e=rng.uniform(-1, 1, (D, 3 * ns, 3 * ns)) / ns))
        ref.append(plans[-1](*arrays).cpu())
    failed = []

    def work(k):
        try:
            with torch.cuda.stream(torch.cuda.Stream()):
                for _ in range(150):
                    out = plans[k](*arrays)
                torch.cuda.current_stream().synchronize()
                assert torch.equal(out.cpu(), ref[k])
        except BaseException as e:  # told to the main thread
            failed.append(e)

    threads = [threading.Thread(target=work, args=(k,)) for k in (0, 1)]
    for th in threads:
        th.start()
    for th in threads:
        th.join()
    assert not failed, failed
