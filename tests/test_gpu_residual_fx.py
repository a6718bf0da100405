"""The FP64 refinement residual in 64-bit fixed point: the ||f - A u|| / ||f||
that a refined solve reports against the oracle's double-double residual of
the same f and u, at the edges of the kernels' tiles (16 x 32 columns by 64
planes in 3D; 30 columns a warp and 2 to 64 rows in 2D), on every kind of face
and element, and for loads whose size changes by many orders inside a tile.
"""
import math

import numpy as np
import pytest
import torch

from oracle import fem
from workloads import ppw_omega, random_rhs

pytestmark = pytest.mark.gpu

SHAPES_2D = [(3, 3), (5, 29), (64, 30), (65, 31), (66, 61), (33, 240), (127, 241), (300, 700), (2100, 1300)]
SHAPES_3D = [(3, 3, 3), (5, 15, 31), (64, 16, 32), (65, 17, 33), (66, 40, 20), (130, 33, 65), (20, 70, 97)]


def load(shape, kind):
    f = random_rhs(shape, 11)
    if kind == "spike":  # one node: quiet tiles beside a loud one
        f[:] = 0
        f[tuple(n // 3 for n in shape)] = 1 + 2j
    elif kind == "ramp":  # grows by 1e12 along x: the tiles' exponents follow
        f *= np.logspace(-12, 0, shape[0]).reshape((-1,) + (1,) * (len(shape) - 1))
    elif kind in ("small", "large"):
        f *= 1e-25 if kind == "small" else 1e25
    return f


def solve(shape, f, bc, elem, tol, max_iter):
    import paper_1809_03808_gb300 as helm

    h = tuple((1.0 + 0.2 * k) / (n - 1) for k, n in enumerate(shape))
    omega = ppw_omega(max(h), 10)
    plan = helm.Plan(shape, h, omega, helm.HELM_C64_REFINED, bc=bc, element=elem)
    helm.helm_set_refinement(plan.handle, tol, max_iter)
    u = plan.solve(torch.from_numpy(f).cuda())
    info, _ = plan.info()
    got = info.residual[info.iterations]
    conv = info.converged
    plan.close()
    return h, omega, u.cpu().numpy(), got, conv


def check(shape, kind, bc, elem, tol):
    f = load(shape, kind)
    h, omega, u, got, _ = solve(shape, f, bc, elem, tol, 10)
    # powers of ten keep the oracle's products in range
    s = 10.0 ** -round(math.log10(np.abs(f).max()))
    r = fem.residual_dd(f * s, u * s, h, omega, bc=bc or "abc", elem=elem)
    r = r[0] if isinstance(r, tuple) else r
    want = np.linalg.norm(r) / np.linalg.norm(f * s)
    # the report: complex64 residuals and their FP32 sums; the arithmetic:
    # coefficients rounded in FP64 (2^-52) and the fixed-point sum (2^-55)
    # of sum |c| max |u|
    top = sum(2.0 / hk for hk in h) + omega ** 2 * max(h)
    csum = top * 4 * math.prod(h) / min(h)  # above sum |c| of any point
    bound = 1e-4 * want + 2.0 ** -50 * csum * np.abs(u * s).max() * math.sqrt(u.size) / np.linalg.norm(f * s)
    assert abs(got - want) <= bound, (got, want, bound)


@pytest.mark.parametrize("shape", SHAPES_2D + SHAPES_3D)
@pytest.mark.parametrize("tol", [1e-4, 1e-14])
def test_tile_edges(shape, tol):
    check(shape, "gaussian", None, "q1", tol)


@pytest.mark.parametrize("shape", [(66, 61), (300, 257), (65, 17, 33), (66, 40, 20)])
@pytest.mark.parametrize("kind", ["spike", "ramp", "small", "large"])
@pytest.mark.parametrize("tol", [1e-4, 1e-14])
def test_ranges(shape, kind, tol):
    check(shape, kind, None, "q1", tol)


@pytest.mark.parametrize("shape", [(66, 61), (65, 17, 33)])
@pytest.mark.parametrize("neumann", [0, 1])
@pytest.mark.parametrize("elem", ["q1", "q1mod"])
def test_faces_and_elements(shape, neumann, elem):
    bc = tuple("neumann" if k == neumann else "abc" for k in range(len(shape)))
    check(shape, "gaussian", bc, elem, 1e-4)


@pytest.mark.parametrize("shape", [(66, 61), (65, 17, 33)])
@pytest.mark.parametrize("bad", [np.nan, np.inf])
def test_not_finite(shape, bad):
    f = load(shape, "gaussian")
    f[tuple(n - 2 for n in shape)] = bad
    _, _, _, got, conv = solve(shape, f, None, "q1", 1e-8, 3)
    assert conv == 0 and not got <= 1e-8
