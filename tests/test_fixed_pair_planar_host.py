"""Fixed point pairs (csrc/fixed_pair.cuh, built for the host) of a plane seen
from just beside it: where every product of a dot product is small, the pair
keeps the accuracy of its products or takes the FP64 form."""
import ctypes
import os
import subprocess

import pytest

HERE = os.path.join(os.path.dirname(os.path.abspath(__file__)), "fixed_pair")
SRC = os.path.join(HERE, "fixed_pair_planar.cpp")


@pytest.fixture(scope="module")
def host(tmp_path_factory):
    out = str(tmp_path_factory.mktemp("fixed_pair") / "libplanar.so")
    subprocess.check_call(["g++", "-O2", "-std=c++17", "-fPIC", "-shared", "-o", out, SRC])
    return ctypes.CDLL(out)


# A dot product is off by at most 11 units of 2^-60 of full scale and, where a coordinate
# is below the grid, by 96 more (half a quantum per coordinate, at the least distance such
# points keep to fixed point); kept products come to 2^50 of these units, so each of the
# two dots is good to 107 / 2^50 = 9.5e-14 of its products.
BOUND = 2 * 107 * 2.0 ** -50 + 8 * 2.0 ** -52


@pytest.mark.parametrize("z0", [0.0, 10.0])
@pytest.mark.parametrize("tilt", [0.0, 1.0])
@pytest.mark.parametrize("h", [30.0, 1.0, 1e-2, 1e-4, 1e-7, 1e-10])
def test_error_against_the_products(host, h, tilt, z0):
    out = (ctypes.c_double * 2)()
    d = ctypes.c_double
    host.planar_errors(20000, d(30.0), d(z0), d(h), d(tilt), out)
    assert out[1] <= BOUND
    if z0 != 0.0 and tilt == 0.0:  # exact coordinates and vectors: no pair needs FP64 but those
        assert out[0] < 20000 // 100  # of points next to x = 0 or y = 0


def test_the_plane_itself_keeps_fixed_point(host):
    """Exactly zero products lose nothing."""
    out = (ctypes.c_double * 2)()
    d = ctypes.c_double
    host.planar_errors(20000, d(30.0), d(0.0), d(0.0), d(1.0), out)
    assert out[1] == 0.0 and out[0] < 20000 // 100
