"""The evaluation kernel's chunks of the last axis (evaluate.cu): one chunk (N + 1 <= 32), the first
size with two, odd counts whose chunk is padded, the smallest N and a large one, 2D and 3D, against
the oracle's direct sum, with the bar of test_gpu_accuracy (1e-12 of the largest value)."""
import numpy as np
import pytest

from oracle import oracle as O

pytestmark = pytest.mark.gpu


@pytest.mark.parametrize("d,N", [(2, 2), (2, 3), (2, 31), (2, 32), (2, 48), (2, 64), (2, 131), (3, 2), (3, 8), (3, 33)])
@pytest.mark.parametrize("r", [0, 1])
def test_evaluate_chunks(d, N, r):
    import torch
    from paper_2105_08806_gb300 import Plan
    rng = np.random.default_rng(N + 1000 * d)
    coef = rng.standard_normal((N + 1) ** d)
    npts = 97
    pts = rng.standard_normal((npts, d)) * 2.5
    out = torch.empty(npts, dtype=torch.float64, device="cuda")
    with Plan(d, N, 4, 2.0, 0.0, 1e-6, map_log=(r == 0)) as plan:
        plan.evaluate(torch.as_tensor(coef, device="cuda"), torch.as_tensor(pts.ravel(), device="cuda"), out)
        torch.cuda.synchronize()
    ref = O.fN_values(coef, d, N, 2.0, r, pts)
    assert np.abs(out.cpu().numpy() - ref).max() <= 1e-12 * np.abs(ref).max()
