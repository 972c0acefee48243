"""Cached graphs tell the two storage layouts of one buffer apart: the same
matrix, vectors, options and workspace solved as n x T and as T x n."""
import pytest

pytestmark = pytest.mark.gpu


# square, and two shapes of one pitch; two-pass products and (2048) the fused pass
@pytest.mark.parametrize("n,T,pitch", [(384, 384, 384), (500, 510, 512), (2048, 2048, 2048)])
@pytest.mark.parametrize("lanczos", [0, 1])
@pytest.mark.parametrize("two_pass", [0, 1])
def test_one_buffer_in_both_layouts(n, T, pitch, lanczos, two_pass):
    import torch

    from paper_2604_02917_gb300 import mv

    g = torch.Generator(device="cuda").manual_seed(n)
    L = torch.randn((max(n, T), pitch), generator=g, device="cuda") * 0.01
    L *= torch.linspace(0.5, 2.0, pitch, device="cuda")          # far from symmetric
    mu = torch.linspace(-1e-3, 1e-3, n, dtype=torch.float64, device="cuda")
    start = torch.randn(n, generator=g, device="cuda", dtype=torch.float64)
    opts = dict(power_start=start, eps=1e-7, max_iter=400, lanczos=lanczos, power_iters=25, two_pass=two_pass)

    def solver(layout):
        rows = L[:n] if layout == "nt" else L[:T]
        return mv.Solver(rows, mu, 2e-4, T, layout=layout, **opts)

    own = {k: solver(k).solve() for k in ("nt", "tn")}            # a workspace each
    assert (own["nt"][0] - own["tn"][0]).abs().max() > 1e-4
    shared = {k: solver(k) for k in ("nt", "tn")}
    ws = torch.empty(max(s.ws.numel() for s in shared.values()), dtype=torch.uint8, device="cuda")
    for k in ("nt", "tn", "nt"):
        shared[k].ws = ws
        x, info = shared[k].solve()
        assert torch.equal(x, own[k][0])
        assert info["iterations"] == own[k][1]["iterations"]
        assert info["lambda_hat"] == own[k][1]["lambda_hat"]
