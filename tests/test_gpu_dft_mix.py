"""The mixed-radix and Bluestein transforms against numpy's FFT in FP64: the
transform of the load that helm_solve_debug returns (eq. step1FFTfcoeff, with
the auxiliary's scaling), for every radix, the primes' own passes, composite
lengths of one to four passes and Bluestein lengths, along the contiguous and
the middle axis."""
import math

import numpy as np
import pytest
import torch

from workloads import random_rhs

pytestmark = pytest.mark.gpu

EPS = {"c64": 2.0 ** -24, "c128": 2.0 ** -53}


def scaled_dft(f, axis, rho, q):
    n = f.shape[axis]
    t = (rho + 0.5j * math.pi * q) / n
    shape = [n if k == axis else 1 for k in range(f.ndim)]
    return np.fft.fft(f * np.exp(-t * np.arange(n)).reshape(shape), axis=axis)


def run(shape, kind):
    import paper_1809_03808_gb300 as helm

    h = [1.0 / (n - 1) for n in shape]
    plan = helm.Plan(shape, h, 2 * math.pi / (10 * max(h)), helm.HELM_C128 if kind == "c128" else helm.HELM_C64_RAW)
    f = random_rhs(shape, 7, np.complex128 if kind == "c128" else np.complex64)
    fd = torch.from_numpy(f).cuda()
    fhat = torch.empty_like(fd)
    helm.helm_solve_debug(plan.handle, fd, torch.empty_like(fd), fhat)
    info, _ = plan.info()
    plan.close()
    want = f.astype(np.complex128)
    for axis in range(1, len(shape)):
        want = scaled_dft(want, axis, info.aux_rho, info.aux_q)
    return np.linalg.norm(fhat.cpu().numpy() - want) / np.linalg.norm(want)


def bound(shape, kind):
    # four roundings per level of a transform there and back (Bluestein) of
    # 2n - 1 points, eight more for the scalings and chirps, every axis
    return EPS[kind] * sum(4 * (2 * math.log2(2 * n) + 8) for n in shape[1:])


ROWS = [3, 5, 6, 7, 9, 10,                                   # one register pass
        11, 13, 17, 19, 43, 59, 61, 34, 129, 17 * 16, 61 * 61,  # the primes' passes: alone, first, twice
        12, 14, 15, 18, 21, 77, 143, 169, 240, 255, 1000, 1001, 1155, 2310, 4095,  # two to five passes
        67, 127, 134, 223, 509, 1021, 2039]                  # Bluestein


@pytest.mark.parametrize("kind", ["c64", "c128"])
@pytest.mark.parametrize("n", ROWS)
def test_rows(n, kind):
    shape = (5, n)
    assert run(shape, kind) <= bound(shape, kind)


@pytest.mark.parametrize("n", [8190, 6561, 4093])
def test_long_rows_c64(n):
    shape = (3, n)
    assert run(shape, "c64") <= bound(shape, "c64")


# many lines: several lines a CTA, a ragged last CTA
@pytest.mark.parametrize("kind", ["c64", "c128"])
@pytest.mark.parametrize("shape", [(2051, 9), (1300, 150), (1111, 67), (999, 43)])
def test_many_rows(shape, kind):
    assert run(shape, kind) <= bound(shape, kind)


@pytest.mark.parametrize("kind", ["c64", "c128"])
@pytest.mark.parametrize("shape", [(3, 3, 3), (3, 15, 17), (4, 43, 5), (3, 150, 33), (3, 1000, 18), (3, 129, 61),
                                   (3, 1021, 9), (5, 67, 127), (40, 80, 72), (3, 34, 1023), (70, 223, 36)])
def test_columns(shape, kind):
    assert run(shape, kind) <= bound(shape, kind)
