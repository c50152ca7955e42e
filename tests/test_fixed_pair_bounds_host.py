"""The bounds csrc/fixed_pair.cuh states for the parts of a pair, built for the host,
against quadruple precision."""
import ctypes
import os
import subprocess

import pytest

HERE = os.path.join(os.path.dirname(os.path.abspath(__file__)), "fixed_pair")
SRC = os.path.join(HERE, "fixed_pair_bounds.cpp")


@pytest.fixture(scope="module")
def host(tmp_path_factory):
    out = str(tmp_path_factory.mktemp("fixed_pair") / "libbounds.so")
    subprocess.check_call(["g++", "-O2", "-std=c++17", "-fPIC", "-shared", "-o", out, SRC])
    return ctypes.CDLL(out)


# Dot product: three dropped low x low products and the floor of the cross sum, each less than a
# unit and all one way; three limbs of the difference cut below a unit and three of the vector
# rounded by half of one, times at most 1.  1/r: W loses four units likewise and twice three cut
# limbs, of at least 2^58, halved by the root, beside fx_rsqrt's 2^-58.  Conversion: truncation.
@pytest.mark.parametrize("sep", [2.0, 0.5, 1e-3])
@pytest.mark.parametrize("span", [0, 4, 40])
def test_bounds(host, sep, span):
    out = (ctypes.c_double * 4)()
    host.bounds(200000, ctypes.c_double(sep), span, out)
    low, high, rinv, conv = out
    assert -8.5 < low and high < 4.5
    assert rinv < 5 * 2.0 ** -58 + 2.0 ** -58
    assert conv < 2.0 ** -52
