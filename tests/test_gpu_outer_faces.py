"""The outer face reduction and face operator of 3D solves at the edges of
their splits (four threads per output with batches of 8 modes; one thread from
155,648 outputs on) and of the 3 x 3 stencil, against the oracle."""
import numpy as np
import pytest
import torch

from oracle import solvers
from workloads import ppw_omega, random_rhs

pytestmark = pytest.mark.gpu

SHAPES = [(3, 3, 3), (5, 4, 6), (4, 5, 3), (6, 31, 5), (5, 32, 4), (9, 33, 7), (4, 35, 16), (16, 64, 17), (5, 257, 6),
          (64, 6, 65), (380, 5, 410)]


@pytest.mark.parametrize("shape", SHAPES)
@pytest.mark.parametrize("mode", ["c128", "c64"])
def test_faces(shape, mode):
    import paper_1809_03808_gb300 as helm

    h = 1.0 / (max(shape) - 1)
    h = (h, 0.9 * h, h)
    omega = ppw_omega(max(h), 9)
    f = random_rhs(shape, 11)
    want, _ = solvers.oracle_solve(f, h, omega, method="tensor")
    plan = helm.Plan(shape, h, omega, helm.HELM_C128 if mode == "c128" else helm.HELM_C64_REFINED)
    u = plan.solve(torch.from_numpy(f).to("cuda")).cpu().numpy()
    plan.close()
    err = np.linalg.norm(u - want) / np.linalg.norm(want)
    assert err <= 1e-10, err  # the parity bound of the other 3D tests
