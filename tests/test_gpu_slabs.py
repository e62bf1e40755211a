"""FP32 spreading in slabs (spread_impl.cuh: slab_range, half quads in 2D, points by size in 3D) on
grids that oversampling 4 makes too large for one block, both maps, with and without an angular
factor, against the FP64 path at the default oversampling.  The transform's error is 0.2-8 tol of the
gain norm and FP32 rounding about 1e-6 of it (test_gpu_kernel_widths, test_gpu_parity), so plans of
tol 1e-7 stay within 5e-6 of the gain norm; a point lost or counted twice at a slab's edge costs far
more."""
import numpy as np
import pytest

from oracle import oracle as O
from paper_2105_08806_gb300 import PG_PREC_FP32, PG_PREC_FP64
from paper_2105_08806_gb300 import workloads as W

from _helpers import gpu_collide

pytestmark = pytest.mark.gpu


@pytest.mark.parametrize("log", [False, True])
@pytest.mark.parametrize("d,N,M,ang", [(2, 61, 6, None), (2, 64, 8, [1.0, 0.4, 0.3]), (3, 10, 6, None),
                                       (3, 11, 4, [1.0, 0.0, 0.5])])
def test_slabs_match_fp64(d, N, M, ang, log):
    S, gamma = 2.5, 0.5
    c = np.array([0.7, -0.4, 0.2])[:d]
    f = lambda p: W.maxwellian(p, 0.6, c, 0.8) + W.maxwellian(p, 0.4, -c, 1.2)  # noqa: E731
    ft = O.project(f, d, N, S, 0 if log else 1).ravel()
    ref, _, mom = gpu_collide(ft, d, N, M, S, gamma, 1e-12, precision=PG_PREC_FP64, map_log=log, angular=ang)
    Q, info, _ = gpu_collide(ft, d, N, M, S, gamma, 1e-7, precision=PG_PREC_FP32, map_log=log, angular=ang, upsampfac=4.0)
    assert info["slabs"] >= 2
    assert np.linalg.norm(Q - ref) < 5e-6 * mom["norm_gain"]
