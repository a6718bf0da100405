"""The 2D chunk carries, face sums and face operator at the edges of their
blocks against the oracle: chunks of 8 (complex128) and 16 (complex64) rows,
segments of at least 4 chunks and at most 32 of them, 8 or 16 lines per carry
block, 32 or 128 lines per face partial, 30 rows per block of the face operator;
and of the one-launch steps: 2, 4 or 8 lines per block, up to 512 threads."""
import numpy as np
import pytest
import torch

from oracle import solvers
from workloads import ppw_omega, random_rhs

pytestmark = pytest.mark.gpu

SHAPES = [(3, 4), (8, 16), (9, 33), (30, 17), (31, 32), (32, 31), (33, 15), (61, 129), (64, 48), (65, 30), (129, 34),
          (513, 20), (1025, 18), (1040, 33), (2049, 16), (2433, 385),
          # one launch per step: the last line lengths of 2 and 4 lines per block, more lines per block, 64 partials
          (2048, 6), (1024, 607), (1025, 610), (128, 255), (136, 256), (47, 1217), (3, 1210)]


@pytest.mark.parametrize("shape", SHAPES)
def test_edges(shape):
    import paper_1809_03808_gb300 as helm

    h = (1.0 / (shape[0] - 1), 1.1 / (shape[0] - 1))
    omega = ppw_omega(max(h), 12)
    f = random_rhs(shape, 7)
    want, _ = solvers.oracle_solve(f, h, omega, method="tensor")
    fd = torch.from_numpy(f).to("cuda")
    for mode in (helm.HELM_C128, helm.HELM_C64_REFINED):
        plan = helm.Plan(shape, h, omega, mode)
        u = plan.solve(fd).cpu().numpy()
        plan.close()
        err = np.linalg.norm(u - want) / np.linalg.norm(want)
        assert err <= 1e-10, (mode, err)  # the parity bound of the other 2D tests
