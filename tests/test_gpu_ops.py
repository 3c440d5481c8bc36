"""A level's products as the solver launches them: the deep-interior fast paths
(FP64 constant viscosity: from 2^19 cells up) against the general rows, and the
product with its inner product in column strips against the product alone, bit
for bit. Sizes around a strip's 60 columns, at each number of rows that a warp
walks (1, 2, 4, 8), the smallest levels that take the strips and ones just
below, odd sides, natural sides; viscosity per cell in FP32."""
import ctypes
import os
import subprocess

import pytest

from paper_2001_10424_gb300 import build

pytestmark = pytest.mark.gpu

HERE = os.path.dirname(os.path.abspath(__file__))
D, N = 0, 1


@pytest.fixture(scope="module")
def probe(lib, tmp_path_factory):
    out = str(tmp_path_factory.mktemp("ops") / "probe.so")
    subprocess.run([build.nvcc_path()] + build.ARCH + build.FLAGS +
                   ["-I", build.CSRC, "-I", os.path.join(os.path.dirname(HERE), "include"), "-cudart", "static", "-shared",
                    "-o", out, os.path.join(HERE, "ops_probe.cu"), build.LIB, "-Xlinker", "-rpath",
                    "-Xlinker", os.path.dirname(build.LIB)], check=True)
    return ctypes.CDLL(out).probe


@pytest.mark.parametrize("mode", [0, 1])
@pytest.mark.parametrize("prec,n,bc,var", [
    (32, (48, 2731), (D,) * 4, 0), (32, (47, 2900), (D,) * 4, 0), (32, (60, 2185), (D, N, N, D), 0),
    (32, (61, 2150), (N, D, D, N), 0), (32, (62, 2115), (D,) * 4, 1), (32, (181, 725), (N, N, N, N), 1),
    (32, (363, 362), (D, N, D, D), 0), (32, (601, 480), (D,) * 4, 1), (32, (1021, 515), (D, D, N, D), 0),
    (32, (1023, 1031), (D,) * 4, 0), (32, (1023, 1031), (D, N, D, N), 1), (32, (2048, 515), (D,) * 4, 0),
    (64, (48, 5462), (D,) * 4, 0), (64, (61, 4300), (N, D, D, N), 0), (64, (541, 485), (D, N, N, D), 0),
    (64, (511, 512), (D,) * 4, 0), (64, (724, 723), (D,) * 4, 0), (64, (725, 724), (D, N, N, N), 0),
    (64, (1023, 1031), (D, D, D, N), 0)])
def test_products_of_a_level(probe, prec, n, bc, var, mode):
    sides = (ctypes.c_int * 3)(n[0], n[1], 1)
    nat = (ctypes.c_int * 6)(*bc, 0, 0)
    diff, dot = (ctypes.c_longlong * 2)(-1, -1), ctypes.c_double(-1)
    assert probe(int(prec == 64), sides, nat, var, mode, diff, ctypes.byref(dot)) == 0
    assert list(diff) == [0, 0]
    # FP64 sums of about 1e6 products: each of the two orders' partial sums
    # rounds to 2^-53 of the sum of absolute products, a few thousand times
    assert 0 <= dot.value <= 1e-12
