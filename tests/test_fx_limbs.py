"""The fixed-point residual's coefficients as 32-bit limbs (csrc/helm_fx.h):
every pair the kernels multiply by is its coefficient rounded to the common
scale, the negated imaginary parts among them, also where the low limb is
-2^31 and so has no 32-bit negative."""
import ctypes
import math
import os
import subprocess

import numpy as np
import pytest

from paper_1809_03808_gb300 import _build

SHIM = """
#include "helm_fx.h"
extern "C" void limbs(double re, double im, int es, int* out) {
  const helm::LimbC c = helm::fx_limb_c(re, im, es);
  const helm::Limb l[3] = {c.re, c.im, c.nim};
  for (int k = 0; k < 3; ++k) { out[2 * k] = l[k].h; out[2 * k + 1] = l[k].l; }
}
"""


@pytest.fixture(scope="module")
def limbs(tmp_path_factory):
    d = tmp_path_factory.mktemp("fx")
    (d / "shim.cpp").write_text(SHIM)
    so = str(d / "shim.so")
    subprocess.run([os.environ.get("CXX", "g++"), "-O2", "-std=c++17", "-I" + _build.CSRC, "-fPIC", "-shared",
                    str(d / "shim.cpp"), "-o", so], check=True)
    f = ctypes.CDLL(so).limbs
    f.argtypes = [ctypes.c_double, ctypes.c_double, ctypes.c_int, ctypes.c_void_p]
    f.restype = None

    def call(re, im, es):
        out = np.zeros(6, dtype=np.int32)
        f(re, im, es, out.ctypes.data)
        return [(int(h) << 32) + int(l) for h, l in out.reshape(3, 2)], [int(l) for l in out[1::2]]

    return call


# a wave number in FP32 on dyadic spacings (129 points, modified elements) has
# face coefficients with a low limb of -2^31: -0.0208... at eS = 3
@pytest.mark.parametrize("omega", [31.9526309967041, 31.83878517150879])
def test_single_precision_wave_numbers(limbs, omega):
    im = -omega * (1.0 / 128.0) / 12.0
    vals, low = limbs(im, im, 3)
    assert -2 ** 31 in low
    c = round(math.ldexp(im, 59))
    assert vals == [c, c, -c]


@pytest.mark.parametrize("es", [-3, 0, 5])
def test_limbs_reproduce_the_coefficient(limbs, es):
    rng = np.random.default_rng(7)
    c = [0, 1, -1, 2 ** 31, -2 ** 31, 2 ** 31 - 1, 2 ** 62, -2 ** 62, 3 * 2 ** 31, -3 * 2 ** 31, 5 * 2 ** 40 + 2 ** 31]
    c += [int(x) << 31 for x in rng.integers(-2 ** 30, 2 ** 30, 200)]  # low limbs 0 and -2^31
    c += [int(x) for x in rng.integers(-2 ** 52, 2 ** 52, 200)]
    for a, b in zip(c, c[1:] + c[:1]):
        vals, _ = limbs(math.ldexp(a, es - 62), math.ldexp(b, es - 62), es)
        assert vals == [a, b, -b]


def test_not_finite(limbs):
    assert limbs(math.inf, math.nan, 2)[0] == [0, 0, 0]
