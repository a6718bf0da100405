"""The tiled inner sweeps of 3D solves at the edges of their chunks (8, 16 and
32 rows), batches (8 rows), staged pivot rows (the first 20, the last 8) and
tiles (16 modes; 16-byte copies need an even number of modes), in every launch
shape (up to 256, 512 and 1024 threads), against the oracle."""
import numpy as np
import pytest
import torch

from oracle import solvers
from workloads import ppw_omega, random_rhs

pytestmark = pytest.mark.gpu

SHAPES = [(3, 4, 16), (9, 5, 3), (17, 4, 31), (20, 3, 32), (29, 5, 18), (33, 4, 17), (64, 3, 16), (65, 4, 34),
          (127, 3, 20), (256, 3, 16), (257, 4, 18), (300, 3, 33), (513, 3, 16), (700, 3, 20), (1030, 3, 18)]


@pytest.mark.parametrize("shape", SHAPES)
@pytest.mark.parametrize("mode", ["c128", "c64"])
def test_chunks(shape, mode):
    import paper_1809_03808_gb300 as helm

    # a long thin box: the x lines run from propagating to evanescent
    h = (1.0 / (shape[0] - 1), 1.0 / (shape[0] - 1), 0.8 / (shape[0] - 1))
    omega = ppw_omega(max(h), 9)
    f = random_rhs(shape, 5)
    want, _ = solvers.oracle_solve(f, h, omega, method="tensor")
    plan = helm.Plan(shape, h, omega, helm.HELM_C128 if mode == "c128" else helm.HELM_C64_RAW)
    fd = torch.from_numpy(f).to("cuda", torch.complex128 if mode == "c128" else torch.complex64)
    tol = 1e-10 if mode == "c128" else 1e-4  # the parity bounds of the other 3D tests
    ran = 0
    for ch in (0, 8, 16, 32):  # 0: the plan's own choice
        if ch:
            try:
                helm.helm_set_variant(plan.handle, helm.HELM_VARIANT_INNER_CHUNK, ch)
            except helm.HelmError:  # too many chunks for one CTA
                continue
        u = plan.solve(fd).cpu().numpy().astype(np.complex128)
        err = np.linalg.norm(u - want) / np.linalg.norm(want)
        assert err <= tol, (ch, err)
        ran += 1
    plan.close()
    assert ran >= 1
