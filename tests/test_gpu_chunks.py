"""The solve loop launches a chunk ahead only where it will be needed: a solve
that ends in its first or second chunk runs no empty one behind it."""
import numpy as np
import pytest

torch = pytest.importorskip("torch")

from synth import CFG_SMALL, factor_returns, power_start

pytestmark = pytest.mark.gpu
CHUNK = 10


def problem(n=200, T=1000):
    from paper_2604_02917_gb300 import mv

    R = torch.from_numpy(factor_returns(CFG_SMALL.scaled(n, T, seed=5), np.float32)).cuda()
    L, _, mu, _ = mv.center_factor(R, "f32")
    opts = dict(power_start=torch.from_numpy(power_start(n)).cuda(), eps=1e-6, two_pass=1)
    return mv, L, mu, float(np.percentile(mu.cpu().numpy(), 60)), T, opts


def test_short_solves_launch_no_empty_chunk():
    mv, L, mu, Rt, T, opts = problem()
    x, info = mv.npga_solve(L, mu, Rt, T, **opts)
    alpha, base = info["alpha"], 4                       # what a solve launches beside its chunks and the objective

    def launches(**kw):
        s = mv.Solver(L, mu, Rt, T, alpha=alpha, kkt_every=CHUNK, **{**opts, **kw})
        return lambda *a: s.solve(*a)[1]

    warm = launches()(x)                                  # stops at its first KKT test
    assert warm["iterations"] == 0 and warm["converged"] == 1
    assert warm["launches"] == base + 3 * CHUNK + 1
    for max_iter, chunks in ((5, 1), (9, 1), (10, 2), (15, 2)):
        info = launches(max_iter=max_iter, eps=0.0)()
        assert info["iterations"] == max_iter
        assert info["launches"] == base + 3 * CHUNK * chunks + 1, max_iter


# the iterates do not depend on how the chunks are launched; ends on and beside a chunk's edge
@pytest.mark.parametrize("max_iter", [0, 1, 19, 20, 21, 40, 57, 10000])
@pytest.mark.parametrize("kkt_every", [10, 0, 3])
def test_same_solution_with_and_without_graphs(max_iter, kkt_every):
    if kkt_every == 0 and max_iter == 10000:
        pytest.skip("no KKT test would end it")
    mv, L, mu, Rt, T, opts = problem()
    got = [mv.npga_solve(L, mu, Rt, T, max_iter=max_iter, kkt_every=kkt_every, use_graph=g, **opts) for g in (1, 0)]
    assert torch.equal(got[0][0], got[1][0])
    for key in ("iterations", "converged", "status", "kkt", "objective"):
        assert got[0][1][key] == got[1][1][key], key
    chunk = kkt_every or 8
    # at most one chunk ahead
    assert 0 <= got[0][1]["launches"] - got[1][1]["launches"] <= 3 * chunk
