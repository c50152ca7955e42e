"""Workspace of the mixed direct sums: what a source split adds is its partial results and
its work items, counted for the tile in use."""
import ctypes

import numpy as np
import pytest

import oracle
from tests._util import cuda, rel_l2

pytestmark = pytest.mark.gpu
# bytes of an item: 512 candidates, frame, item, counts; rounded up to whole 256 bytes by array
ITEM = 512 * 4 + 12 * 4 + 24 + 8 + 16


@pytest.fixture(scope="module")
def lib():
    from paper_1909_11085_gb300 import build
    build.build()
    import paper_1909_11085_gb300 as P
    return P


def _bytes(ns, nt, splits, tile):
    from paper_1909_11085_gb300 import _abi as A
    o, n = A.make_opts("mixed", 1.0, False, splits, tile), ctypes.c_size_t(0)
    A.check(A.lib().stokes_direct_workspace_size(ns, nt, 2, ctypes.byref(o), ctypes.byref(n)))
    return n.value


@pytest.mark.parametrize("nt", [129, 5000, 204800])
def test_bytes_of_a_split(lib, nt):
    a, b = _bytes(139264, nt, 8, 0), _bytes(139264, nt, 40, 0)
    assert b - a <= 32 * (24 * nt + -(-nt // 128) * ITEM) + 16 * 256


@pytest.mark.parametrize("tile", [-1, 0, 1, 2, 3])
@pytest.mark.parametrize("nt", [1, 63, 129, 700])
def test_every_tile_fits_its_own(lib, tile, nt):
    import torch
    from paper_1909_11085_gb300 import _abi as A
    rng = np.random.default_rng(nt)
    ns = 900
    src, trg, phi, nrm = (rng.uniform(-2, 2, (n, 3)) for n in (ns, nt, ns, ns))
    w, h = rng.uniform(0.5, 1.5, ns), np.full(ns, 0.2)
    S, T, P, N, Wt, Hs = cuda(src, trg, phi, nrm, w, h)
    ref = oracle.dl(src, nrm, phi, w, trg)
    for splits in (1, 5):
        o = A.make_opts("mixed", 1.0, False, splits, tile)
        ws, out = A.workspace(_bytes(ns, nt, splits, tile), S.device), torch.empty_like(T)
        A.check(A.lib().stokes_dl_eval(
            A.ptr(S), A.ptr(N), A.ptr(P), A.ptr(Wt), A.ptr(Hs), ns, A.ptr(T), nt, A.ptr(out),
            ctypes.byref(o), A.ptr(ws), ws.numel(), A.stream_ptr(S.device)))
        assert rel_l2(out.cpu().numpy(), ref) <= 1e-6
