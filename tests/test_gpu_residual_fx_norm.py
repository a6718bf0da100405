"""The relative residual a refined solve reports where f is far below the terms
of A u (smooth loads of one sign at hundreds to ten thousand nodes per
wavelength), for f and -f, against the oracle's double-double residual."""
import math

import numpy as np
import pytest
import torch

from oracle import fem
from workloads import ppw_omega

pytestmark = pytest.mark.gpu


@pytest.mark.parametrize("shape", [(129, 129), (1025, 1025), (500, 61), (65, 33, 40)])
@pytest.mark.parametrize("ppw", [200, 10000])
def test_smooth_loads(shape, ppw):
    import paper_1809_03808_gb300 as helm

    h = tuple(1.0 / (n - 1) for n in shape)
    omega = ppw_omega(max(h), ppw)
    x = np.meshgrid(*[np.linspace(0, 1, n) for n in shape], indexing="ij")
    f = (1 + 0.5j) * (1 + 0.1 * np.cos(sum(x)))
    csum = (sum(2.0 / hk for hk in h) + omega ** 2 * max(h)) * 4 * math.prod(h) / min(h)  # above sum |c| of any point
    plan = helm.Plan(shape, h, omega, helm.HELM_C64_REFINED)
    helm.helm_set_refinement(plan.handle, 1.0, 1)  # the residual of the first solve, well above rounding
    got = []
    for sign in (1, -1):
        u = plan.solve(torch.from_numpy(sign * f).cuda())
        info, _ = plan.info()
        got.append(info.residual[info.iterations])
        u = u.cpu().numpy()
        r = fem.residual_dd(sign * f, u, h, omega)
        r = r[0] if isinstance(r, tuple) else r
        want = np.linalg.norm(r) / np.linalg.norm(f)
        # complex64 residuals and FP32 sums of |r|^2 and |f|^2 (1e-4, generous);
        # coefficients and the sum rounded at 2^-50 of sum |c| max |u|
        bound = 1e-4 * want + 2.0 ** -50 * csum * np.abs(u).max() * math.sqrt(u.size) / np.linalg.norm(f)
        assert abs(got[-1] - want) <= bound, (got[-1], want, bound)
    plan.close()
