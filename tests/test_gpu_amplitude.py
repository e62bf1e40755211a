"""FP32 plans over the amplitude of f: Q is quadratic, and a power of two commutes with every rounding,
so Q(s f) = s^2 Q(f) bit for bit as long as nothing leaves FP32's range on the way.  The node values of f
fit it from 1e-38 to 1e38; the products of two of them, their sums and the strength bound do not."""
import numpy as np
import pytest

from oracle import oracle as O
from paper_2105_08806_gb300 import PG_PREC_FP32
from paper_2105_08806_gb300 import workloads as W

pytestmark = pytest.mark.gpu


def _input(d, N):
    c = np.array([0.7, -0.4, 0.2])[:d]
    f = lambda p: W.maxwellian(p, 0.6, c, 0.8) + W.maxwellian(p, 0.4, -c, 1.2)  # noqa: E731
    return O.project(f, d, N, 2.0, 1).ravel()


def _check(collide, f):
    import torch
    f = torch.as_tensor(f, device="cuda")
    Q, Qs = torch.empty_like(f), torch.empty_like(f)
    collide(f, Q)
    for e in (65, 67, 68):  # 3.7e19 .. 3.0e20
        collide(f * 2.0 ** e, Qs)
        torch.cuda.synchronize()
        assert torch.equal(Qs * 2.0 ** (-2 * e), Q), e


@pytest.mark.parametrize("ang", [None, [1.0, 0.5, 0.3]])
@pytest.mark.parametrize("d,N", [(2, 12), (2, 17), (3, 6)])
def test_large_amplitudes(d, N, ang):
    from paper_2105_08806_gb300 import Plan
    with Plan(d, N, 6, 2.0, 0.5, 1e-6, precision=PG_PREC_FP32, angular=ang) as plan:
        _check(plan.collide, _input(d, N))


@pytest.mark.parametrize("d,N", [(2, 12), (3, 6)])
def test_large_amplitudes_batched(d, N):
    from paper_2105_08806_gb300 import BatchedPlan
    with BatchedPlan(d, [N, N], [6, 8], [2.0, 2.0], [0.5, 1.0], 1e-6, precision=PG_PREC_FP32) as plan:
        plan.use_graph(False)
        _check(plan.collide, np.tile(_input(d, N), 2))
