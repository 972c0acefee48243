"""tr(Sigma) of mv_center_factor is as accurate as sums of FP64 squares."""
from fractions import Fraction

import numpy as np
import pytest

pytestmark = pytest.mark.gpu

# T = 987 and 969: 1 / sqrt(T - 1) as a pair of FP32 values is off by 2^-49 (of
# either sign), which alone would make 3.5e-15 of the trace.  The last two are
# below and just above the 2^16 entries from which squares are summed as pairs.
SHAPES = [(300, 987), (300, 969), (1300, 987), (40, 5000), (3, 40), (67, 977), (68, 977)]


def exact_sum_of_squares(R, mu):
    """sum (R_it - mu_i)^2 without rounding: every value is an integer times 2^-120."""
    total = 0
    for row, m in zip(R, mu):
        mi = int(Fraction(float(m)) * (1 << 120))
        v = [int(Fraction(float(x)) * (1 << 120)) - mi for x in row]
        total += sum(u * u for u in v)
    return Fraction(total, 1 << 240)


@pytest.mark.parametrize("shape", SHAPES)
@pytest.mark.parametrize("layout", ["nt", "tn"])
@pytest.mark.parametrize("dt", ["f32", "bf16", "fp8"])
def test_trace_error(shape, layout, dt):
    import torch

    from paper_2604_02917_gb300 import mv

    n, T = shape
    g = np.random.default_rng(n + T)
    R = (g.standard_normal((n, T)) * 0.02 + 3e-4).astype(np.float32)
    _, _, mu, tr = mv.center_factor(torch.from_numpy(R).cuda(), dt, layout=layout)
    exact = exact_sum_of_squares(R, mu.cpu().numpy()) / (T - 1)
    err = float(abs(Fraction(float(tr)) - exact) / exact)
    # Rounding to nearest in an addition tree: the level with 2^k partial sums
    # contributes 2^-53 / sqrt(3) / 2^(k/2) (root mean square), all levels together
    # 2.2e-16 at most with the division by T - 1; the squares average to less.
    # Five times that.
    assert err <= 1.1e-15
