"""The fixed-point residual's face rows at coefficients whose low limb is
-2^31 (wave numbers rounded to FP32 on dyadic spacings), with absorbing faces
and with Neumann faces on one axis: the refined solution against the oracle's,
and the residual it reports against the double-double one."""
import math

import numpy as np
import pytest
import torch

from oracle import fem, solvers
from workloads import random_rhs

pytestmark = pytest.mark.gpu


@pytest.mark.parametrize("neumann", [None, 0, 1])
@pytest.mark.parametrize("shape,omega,elem", [
    ((129, 129), 31.9526309967041, "q1mod"), ((257, 257), 63.9052619934082, "q1mod"),
    ((33, 33, 33), 32.1185188293457, "q1mod"), ((33, 33, 33), 7.881690502166748, "q1")])
def test_low_limb_without_a_negative(shape, omega, elem, neumann):
    import paper_1809_03808_gb300 as helm

    assert float(np.float32(omega)) == omega
    h = tuple(1.0 / (n - 1) for n in shape)
    f = random_rhs(shape, 5)
    bc = tuple("neumann" if k == neumann else "abc" for k in range(len(shape)))
    plan = helm.Plan(shape, h, omega, helm.HELM_C64_REFINED, bc=bc, element=elem)
    helm.helm_set_refinement(plan.handle, 1e-14, 10)
    u = plan.solve(torch.from_numpy(f).cuda()).cpu().numpy()
    info, _ = plan.info()
    got = info.residual[info.iterations]
    plan.close()
    ref, _ = solvers.oracle_solve(f, h, omega, bc=bc, elem=elem)
    # the refinement ends at the residual's rounding (below 1e-14 of |f| here)
    # times the problem's condition (some hundreds)
    assert np.linalg.norm(u - ref) <= 1e-10 * np.linalg.norm(ref)
    r = fem.residual_dd(f, u, h, omega, bc=bc, elem=elem)
    r = r[0] if isinstance(r, tuple) else r
    want = np.linalg.norm(r) / np.linalg.norm(f)
    # complex64 residuals and their FP32 sums; coefficients and sums to 2^-50
    # of sum |c| max |u|
    csum = (sum(2.0 / hk for hk in h) + omega ** 2 * max(h)) * 4 * math.prod(h) / min(h)
    assert abs(got - want) <= 1e-4 * want + 2.0 ** -50 * csum * np.abs(u).max() * math.sqrt(u.size) / np.linalg.norm(f)
