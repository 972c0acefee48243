"""The sketch GEMM's last wave as quarter tiles: 256 x 256 tiles that fill
less than half a wave of 76 CTA pairs, exactly half of the last one, one tile
more than half, one tile into a wave and a whole wave, with edge tiles whose
outer quarters lie outside the product, against FP64 on the stored factor.

Tolerance: FP32 sums of chunks of 256 terms and of the chunk partials, below
1e-5 of the sum of |terms| (a few units of 2^-24 each); FP32 factors add the
two-piece split's 2^-18 per term (4e-6), still below 1e-5.
"""
import pytest

torch = pytest.importorskip("torch")

pytestmark = pytest.mark.gpu


# tiles of 256 x 256: 15, 114 = 76 + 38, 115 = 76 + 39, 77 = 76 + 1, 76
@pytest.mark.parametrize("n,m", [(1100, 700), (19 * 256 - 130, 6 * 256 - 129), (5 * 256 - 1, 23 * 256 - 200),
                                 (11 * 256 - 128, 7 * 256 - 3), (4 * 256, 19 * 256)])
@pytest.mark.parametrize("dt,T", [("bf16", 700), ("f32", 190), ("fp8", 321)])
def test_sketch_last_wave(n, m, dt, T):
    if not torch.cuda.is_available():
        pytest.skip("no CUDA device")
    from paper_2604_02917_gb300 import mv
    g = torch.Generator("cuda").manual_seed(n + m)
    R = torch.randn(n, T, device="cuda", generator=g)
    Phi = mv.bf16_rows(torch.randn(m, T, device="cuda", generator=g))
    L, rs, _, _ = mv.center_factor(R, dt)
    got = mv.sketch_dtype(L, T, Phi, dt, rs).double()
    A = L[:, :T].view(torch.float8_e4m3fn).float().double() * rs.double()[:, None] if dt == "fp8" else L[:, :T].double()
    B = Phi[:, :T].double()
    assert bool(((got - A @ B.T).abs() <= 1e-5 * (A.abs() @ B.abs().T) + 1e-30).all())
