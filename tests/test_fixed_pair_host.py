"""The fixed point pair of the FP64 engine (csrc/fixed_pair.cuh), built for the
host: its error against extended precision beside that of the same pair in
FP64, over kinds, scales, offsets, separations and degenerate vectors."""
import ctypes
import os
import subprocess

import pytest

HERE = os.path.join(os.path.dirname(os.path.abspath(__file__)), "fixed_pair")
SRC = os.path.join(HERE, "fixed_pair_harness.cpp")
HDR = os.path.join(HERE, "..", "..", "paper_1909_11085_gb300", "csrc", "fixed_pair.cuh")


@pytest.fixture(scope="module")
def host():
    out = os.path.join(HERE, "_build", "libfixedpair.so")
    if not os.path.exists(out) or os.path.getmtime(out) < max(os.path.getmtime(SRC),
                                                              os.path.getmtime(HDR)):
        os.makedirs(os.path.dirname(out), exist_ok=True)
        tmp = out + f".tmp{os.getpid()}"
        subprocess.check_call(["g++", "-O2", "-std=c++17", "-fPIC", "-shared", "-o", tmp, SRC])
        os.replace(tmp, out)
    L = ctypes.CDLL(out)
    L.fixed_rsqrt_error.restype = ctypes.c_double
    return L


@pytest.mark.parametrize("kind", [1, 2, 3])
@pytest.mark.parametrize("size,shift,sep", [(50.0, 0.0, 0.0), (50.0, 3.0e3, 0.0), (50.0, 0.0, 1.0),
                                            (50.0, -1e-5, 1e-3), (1e-30, 0.0, 0.0),
                                            (1e30, 0.0, 0.0)])
@pytest.mark.parametrize("planar", [0, 1])
def test_error_is_no_larger_than_fp64s(host, kind, size, shift, sep, planar):
    out = (ctypes.c_double * 5)()
    d = ctypes.c_double
    host.fixed_pair_errors(kind, 20000, d(size), d(shift), d(sep), planar, out)
    slow, rms, worst, rms64, worst64 = out
    assert slow < 20000 // 100
    if kind == 2 and planar:
        assert worst == 0.0  # (d.n) is exactly zero
    # the fixed form's dots and 1/r are good to 2^-58 before they are rounded,
    # so it keeps only the roundings of the products both forms share
    assert rms <= rms64 and worst <= 1.5 * worst64 + 2.0 ** -52


@pytest.mark.parametrize("sep", [1e-9, 0.0])
def test_pairs_below_the_grid_take_fp64(host, sep):
    """Half-width 50: the grid's quantum is 2^-56, pairs closer than 2^-24 go to FP64."""
    out = (ctypes.c_double * 5)()
    d = ctypes.c_double
    host.fixed_pair_errors(3, 1000, d(50.0), d(0.0), d(sep if sep else 1e-300), 0, out)
    assert out[0] == 1000


def test_rsqrt(host):
    assert host.fixed_rsqrt_error(200000) < 2.0 ** -58


@pytest.mark.parametrize("E", [-200, -3, 0, 7, 200])
def test_coordinates(host, E):
    worst = ctypes.c_double()
    assert host.fixed_coord_check(20000, E, ctypes.byref(worst)) == 0
    assert worst.value <= 0.5
