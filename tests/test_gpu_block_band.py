"""FP32 plans whose grid just fits one block: two slabs with full blocks, not one with a few warps (host.cu:
spread_shape), and the FP64 result within test_gpu_slabs' bar for tol 1e-7 (5e-6 of the gain norm)."""
import numpy as np
import pytest

from oracle import oracle as O
from paper_2105_08806_gb300 import PG_PREC_FP32, PG_PREC_FP64
from paper_2105_08806_gb300 import workloads as W

from _helpers import gpu_collide

pytestmark = pytest.mark.gpu


@pytest.mark.parametrize("d,N,M,ang,slabs", [(2, 113, 4, None, 1), (2, 116, 6, None, 2), (2, 117, 4, None, 2),
                                             (2, 115, 4, [1.0, 0.4, 0.3], 2), (3, 16, 4, None, 1), (3, 17, 4, None, 2)])
def test_grids_at_the_edge_of_one_block(d, N, M, ang, slabs):
    S, gamma = 2.5, 0.5
    c = np.array([0.7, -0.4, 0.2])[:d]
    f = lambda p: W.maxwellian(p, 0.6, c, 0.8) + W.maxwellian(p, 0.4, -c, 1.2)  # noqa: E731
    ft = O.project(f, d, N, S, 1).ravel()
    ref, _, mom = gpu_collide(ft, d, N, M, S, gamma, 1e-11, precision=PG_PREC_FP64, angular=ang)
    Q, info, _ = gpu_collide(ft, d, N, M, S, gamma, 1e-7, precision=PG_PREC_FP32, angular=ang)
    assert info["slabs"] == slabs and info["spread_threads"] >= 320
    assert np.linalg.norm(Q - ref) < 5e-6 * mom["norm_gain"]
