"""The loss sums of 2D angular FP32 plans keep the FP64 node values (in two FP32 terms).  With
b = 1 and gamma = 0 every pair term is exactly a_j, so the loss's total mass, the gain's less Q's, is that of the
FP64 plan to rounding (2^-48 of a term: below 1e-12 of the gain's mass; values rounded to FP32 leave 1e-10)."""
import numpy as np
import pytest

from oracle import oracle as O
from paper_2105_08806_gb300 import PG_PREC_FP32, PG_PREC_FP64
from paper_2105_08806_gb300 import workloads as W

from _helpers import gpu_collide

pytestmark = pytest.mark.gpu


@pytest.mark.parametrize("N,M", [(9, 6), (16, 8), (33, 4)])
def test_loss_keeps_the_fp64_node_values(N, M):
    f = lambda p: W.maxwellian(p, 0.6, [0.9, -0.3], 0.7) + W.maxwellian(p, 0.4, [-0.2, 1.1], 1.3)  # noqa: E731
    ft = O.project(f, 2, N, 2.0, 1).ravel()
    loss = []
    for prec, tol in ((PG_PREC_FP32, 1e-6), (PG_PREC_FP64, 1e-12)):
        _, _, mom = gpu_collide(ft, 2, N, M, 2.0, 0.0, tol, precision=prec, angular=[1.0])
        loss.append(mom["mass_gain"] - mom["mass"])
    assert abs(loss[0] - loss[1]) <= 1e-12 * abs(loss[1])
