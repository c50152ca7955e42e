"""FP64 sums of few points, which are bound by their launches: at the lines where the plain
form and the one-block packing end, against the oracle, and the number of launches."""
import numpy as np
import pytest

import oracle
from tests._util import cuda, rel_l2

pytestmark = pytest.mark.gpu
TOL64, GRAD64 = 1e-12, 1e-11


@pytest.fixture(scope="module")
def lib():
    from paper_1909_11085_gb300 import build
    build.build()
    import paper_1909_11085_gb300 as P
    return P


def _counted(call):
    from paper_1909_11085_gb300 import _abi as A
    call()
    n = A.lib().stokes_launch_count()
    out = call()
    return out, A.lib().stokes_launch_count() - n


@pytest.mark.parametrize("ns,nt", [(1, 1), (24, 24), (25, 24), (1, 577), (577, 1), (255, 257),
                                   (256, 257), (512, 0), (513, 0)])
@pytest.mark.parametrize("far", [False, True])
def test_sums(lib, ns, nt, far):
    rng = np.random.default_rng(ns + 1000 * nt)
    src = rng.uniform(-1, 1, (ns, 3)) * (1e-9 if far else 1.0)
    if far:
        src[0] = 1e3  # most sources below the grid: the plain form
    trg = rng.uniform(-1, 1, (nt, 3)) if nt else None
    f, phi, nrm = (rng.uniform(-1, 1, (ns, 3)) for _ in range(3))
    w = rng.uniform(0.5, 1.5, ns)
    S, F, P, N, Wt = cuda(src, f, phi, nrm, w)
    T = cuda(trg)[0] if nt else None
    at = trg if nt else src
    got, launches = _counted(lambda: lib.sldl(S, F, N, P, Wt, T, 0.7, precision="fp64"))
    ref = oracle.sldl(src, f, nrm, phi, w, at, 0.7)
    if np.abs(ref).max() > 0.0:
        assert rel_l2(got.cpu().numpy(), ref) <= TOL64
    # counters, records, items, engine(s), sum of the splits
    assert launches <= (5 if ns * (nt or ns) <= 576 else 6 if ns + nt <= 512 else 8)


def test_gradients_of_one_pair(lib):
    rng = np.random.default_rng(44)
    src, trg, f, phi, nrm, g = (rng.uniform(-1, 1, (1, 3)) for _ in range(6))
    w = np.ones(1)
    args = cuda(src, f, nrm, phi, w, trg, g)
    got, launches = _counted(lambda: lib.sldl_grad(*args, 0.9, precision="fp64"))
    ref = oracle.sldl_grad(src, f, nrm, phi, w, trg, g, 0.9)
    for k, v in got.items():
        assert rel_l2(v.cpu().numpy(), ref["grad_" + k]) <= GRAD64
    # two packs, two orders' boxes (two launches each) and keys, two passes and their sums
    assert launches <= 12
