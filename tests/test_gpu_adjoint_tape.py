"""The reverse sweep's last segment keeps the states of the forward pass
instead of being run again: one segment that the iterations fill exactly or
only in part, a last segment of one step, a whole number of segments and a
single iteration, against the FP64 adjoint of the same factor, step and start.

Tolerance: a segment's d L is one sum of 12 C BF16 products per entry, at
most an ulp of 2^-24 dropped per 16 of them (C <= 64: 48 ulps), and there are
at most three segments, each added once in FP32; with the inputs' own errors
(each a few ulps) this stays below 200 * 2^-24 = 1.2e-5 only in the worst
case of equal signs, so 1e-5 of the largest entry.
"""
import numpy as np
import pytest

torch = pytest.importorskip("torch")

from synth import CFG_SMALL, factor_returns
from oracle.center import center_factor
from oracle.npga import initial_point
from oracle import adjoint

pytestmark = pytest.mark.gpu
TOL = 1e-5


@pytest.mark.parametrize("K,C", [(1, 1), (1, 8), (40, 64), (40, 40), (41, 20), (60, 20)])
def test_last_segment_from_the_forward_pass(K, C):
    if not torch.cuda.is_available():
        pytest.skip("no CUDA device")
    from paper_2604_02917_gb300 import mv
    n, T = 257, 1203
    R = factor_returns(CFG_SMALL.scaled(n, T, seed=83), np.float32)
    L, _, mu, _ = mv.center_factor(torch.from_numpy(R).cuda(), "f32")
    mu_o = center_factor(R.astype(np.float64))[0]
    Rt = float(np.percentile(mu_o, 60))
    x, info = mv.npga_solve(L, mu, Rt, T, eps=0.0, kkt_every=0, max_iter=K)
    L64 = L[:, :T].double().cpu().numpy()
    x0 = initial_point(mu_o, Rt, "ge")
    _, tape, betas = adjoint.unrolled_forward(L64, 0.0, mu_o, Rt, x0, info["alpha"], K, "ge", record=True)
    gx = np.random.default_rng(7).standard_normal(n)
    dmu, dL, binfo = mv.npga_backward(L, mu, Rt, T, torch.from_numpy(gx).cuda(), K, checkpoint_every=C)
    assert binfo["iterations"] == K
    mub, Lb = adjoint.backward(L64, 0.0, mu_o, info["alpha"], tape, betas, gx)
    for got, ref in ((dmu.cpu().numpy(), mub), (dL[:, :T].double().cpu().numpy(), Lb)):
        assert np.max(np.abs(got - ref)) <= TOL * np.max(np.abs(ref))
