"""The arithmetic that the kernels do in place of CUDA's: a quotient from a
reciprocal computed beforehand, and the conversion of floats by integer
instructions. Both have to give the bits of CUDA's division and conversion."""
import ctypes
import os
import subprocess

import pytest

from paper_2001_10424_gb300 import build

pytestmark = pytest.mark.gpu

HERE = os.path.dirname(os.path.abspath(__file__))


@pytest.fixture(scope="module")
def probe(lib, tmp_path_factory):
    out = str(tmp_path_factory.mktemp("arith") / "probe.so")
    subprocess.run([build.nvcc_path()] + build.ARCH + build.FLAGS +
                   ["-I", build.CSRC, "-I", os.path.join(os.path.dirname(HERE), "include"), "-cudart", "static", "-shared",
                    "-o", out, os.path.join(HERE, "arith_probe.cu")], check=True)
    f = ctypes.CDLL(out).probe
    f.argtypes, f.restype = [ctypes.c_int, ctypes.c_int, ctypes.c_longlong], ctypes.c_longlong
    return f


@pytest.mark.parametrize("kind,n", [(0, 1 << 26), (1, 1 << 28), (2, 1 << 20), (3, 1 << 28)])
def test_quotients_have_the_bits_of_the_division(probe, kind, n):
    assert probe(0, kind, n) == 0


@pytest.mark.parametrize("mixed", [0, 1])
def test_conversions_have_the_bits_of_the_cast(probe, mixed):
    assert probe(1, mixed, 0) == 0
