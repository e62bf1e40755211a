"""pg_boltz_evaluate (evaluate.cu) adds the terms of the highest modes first, as the coefficients of smooth
densities fall with the mode number.  Here mode 0 is 1 and the others of one axis are so small that each is
below half a unit of the sum's last place: added to it one by one they would all be lost (N x 0.9 half
units, 3.9e-15 of the sum at N = 48), added up before it they count.  At a point far out on that axis every
T_k is 1 to 1e-7 or better.  The quotient of the values with and without them is off by at most four
roundings (two sums, two products with the weight) and its own: 5 x 2^-53."""
import math

import numpy as np
import pytest

pytestmark = pytest.mark.gpu


@pytest.mark.parametrize("d,N,axis", [(2, 31, 0), (2, 48, 0), (2, 48, 1), (2, 80, 1), (3, 20, 0), (3, 20, 1), (3, 33, 2)])
def test_small_terms_are_added_first(d, N, axis):
    import torch
    from paper_2105_08806_gb300 import Plan
    lead = math.pi ** (-d / 2)
    half_unit = 2.0 ** (math.floor(math.log2(lead)) - 53)
    coef = np.zeros((2,) + (N + 1,) * d)
    coef[(slice(None),) + (0,) * d] = 1.0
    line = [1] + [0] * d
    line[1 + axis] = slice(1, None)
    coef[tuple(line)] = 0.9 * half_unit / (lead * math.sqrt(2.0))
    pts = np.zeros((1, d))
    pts[0, axis] = 1e6  # xi = 1 - 4.5e-12 at S = 3
    out = []
    with Plan(d, N, 4, 3.0, 0.0, 1e-6) as plan:
        for c in coef:
            o = torch.empty(1, dtype=torch.float64, device="cuda")
            plan.evaluate(torch.as_tensor(c.ravel(), device="cuda"), torch.as_tensor(pts.ravel(), device="cuda"), o)
            torch.cuda.synchronize()
            out.append(float(o[0]))
    want = N * 0.9 * half_unit / lead
    assert want > 10 * 2.0 ** -53
    assert abs(out[1] / out[0] - 1.0 - want) <= 5 * 2.0 ** -53
