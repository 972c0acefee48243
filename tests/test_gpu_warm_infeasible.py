"""A warm start skips the projection that finds a target infeasible, so the
first step does, without an exchange over its cluster: all of its blocks have
to take the step before the stop flag is set."""
import pytest

torch = pytest.importorskip("torch")

pytestmark = pytest.mark.gpu


# one block, 4, 8 and 16; two-pass products and the fused pass
@pytest.mark.parametrize("n,T", [(200, 500), (2000, 500), (4000, 500), (5440, 500), (5440, 4200)])
@pytest.mark.parametrize("mode", ["ge", "eq"])
@pytest.mark.parametrize("kkt_every", [0, 10])
def test_infeasible_target_from_a_warm_start(n, T, mode, kkt_every):
    from paper_2604_02917_gb300 import mv

    g = torch.Generator(device="cuda").manual_seed(n)
    L = torch.randn((n, mv.padded_ld(T, mv.DTYPES["f32"])), generator=g, device="cuda") * 0.01
    mu = torch.linspace(-1e-3, 1e-3, n, dtype=torch.float64, device="cuda")
    s = mv.Solver(L, mu, 2e-3, T, mode=mode, kkt_every=kkt_every, max_iter=30, alpha=1.0)
    for _ in range(20):
        with pytest.raises(mv.MvError) as e:
            s.solve(torch.full((n,), 1.0 / n, dtype=torch.float64, device="cuda"))
        assert e.value.status == mv.MV_ERR_INFEASIBLE
        assert s.x.unique().numel() == 1                   # every block did the same
