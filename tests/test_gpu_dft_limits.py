"""Transforms of the longest lengths that a line's two buffers in shared memory
allow (2 n values of 227 KB: n <= 7264 in complex128, 14528 in complex64),
against numpy's FFT: lengths whose padded lines fit and do not fit, with and
without a prime pass, whose roots fit beside the lines or do not; and the first
lengths past the limit."""
import pytest

from test_gpu_dft_mix import bound, run

pytestmark = pytest.mark.gpu

C128 = [6400, 6426, 6480, 7000, 7200, 7245, 7250, 7260]
C64 = [13600, 13640, 13650, 14000, 14400, 14508, 14518, 14520]


@pytest.mark.parametrize("kind,n", [("c128", n) for n in C128] + [("c64", n) for n in C64])
def test_longest_rows(kind, n):
    assert run((3, n), kind) <= bound((3, n), kind)


@pytest.mark.parametrize("kind,n", [("c128", 7290), ("c128", 7546), ("c64", 14553), ("c64", 15000)])
def test_past_the_limit(kind, n):
    import ctypes

    import paper_1809_03808_gb300 as helm

    h = ctypes.c_void_p()
    dtype = helm.HELM_C128 if kind == "c128" else helm.HELM_C64_RAW
    assert helm.lib.helm_plan_2d(ctypes.byref(h), 3, n, 0.5, 1.0 / (n - 1), 10.0, dtype) == helm.HELM_EUNSUPPORTED
