"""The accumulating inverse transform u += S(r) of refinement at the ends of
the FP32 range: loads of extreme size, an exactly zero load and one whose
solution has zero rows, for power-of-two lines of one and several passes and
for mixed-radix and Bluestein lines, against the complex128 solve."""
import numpy as np
import pytest
import torch

from workloads import ppw_omega, random_rhs

pytestmark = pytest.mark.gpu


@pytest.mark.parametrize("shape", [(9, 8), (9, 16), (12, 32), (17, 512), (9, 60), (9, 67), (6, 10, 16), (7, 9, 20)])
@pytest.mark.parametrize("scale", [0.0, 1e-30, 1.0, 1e30])
def test_scales(shape, scale):
    import paper_1809_03808_gb300 as helm

    h = tuple(1.0 / (shape[0] - 1) for _ in shape)
    omega = ppw_omega(max(h), 10)
    f = torch.from_numpy(random_rhs(shape, 3) * scale).cuda()
    ref = helm.Plan(shape, h, omega, helm.HELM_C128)
    want = ref.solve(f).cpu().numpy()
    ref.close()
    plan = helm.Plan(shape, h, omega, helm.HELM_C64_REFINED)
    got = plan.solve(f).cpu().numpy()
    plan.close()
    if scale == 0.0:
        assert not got.any()
        return
    # both are within the 1e-10 parity bound of the exact solution
    assert np.linalg.norm(got / scale - want / scale) <= 2e-10 * np.linalg.norm(want / scale)
