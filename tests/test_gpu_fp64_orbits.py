"""FP64 2D spreading by quads of mirrored classes (spread_impl.cuh: spread_orbits) against the FP64
oracle at the sizes where its numbering can go wrong: even and odd N (an odd N has nodes that are
their own mirror image), M a multiple of 4 or not, both maps, angular kernels, a density without
any symmetry, and the smallest N.  The bar is the FP64 path's (test_gpu_parity): 1e-10 of Q."""
import numpy as np
import pytest

from oracle import oracle as O
from paper_2105_08806_gb300 import PG_PREC_FP64
from paper_2105_08806_gb300 import workloads as W

from _helpers import gpu_collide, rel_l2

pytestmark = pytest.mark.gpu


@pytest.mark.parametrize("N,M,log,ang", [(2, 2, False, None), (3, 4, False, None), (4, 6, True, None), (7, 10, False, None),
                                         (8, 12, True, [1.0, 0.5, 0.3]), (9, 14, False, [0.7, 0.0, 0.6]),
                                         (13, 8, False, None)])
def test_orbits_match_oracle(N, M, log, ang):
    d, S, gamma, r = 2, 2.0, 0.5, 0 if log else 1
    f = lambda p: W.maxwellian(p, 0.6, [0.9, -0.3], 0.7) + W.maxwellian(p, 0.4, [-0.2, 1.1], 1.3)  # noqa: E731
    ft = O.project(f, d, N, S, r).ravel()
    gain, loss = O.collide_parts(ft, d, N, M, S, gamma, r=r, **({"angular": ang} if ang else {}))
    Q, _, _ = gpu_collide(ft, d, N, M, S, gamma, 1e-13, precision=PG_PREC_FP64, map_log=log, angular=ang)
    assert rel_l2(Q, gain - loss) < 1e-10
