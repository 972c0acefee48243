"""The explicit covariance on CTA pairs: 256 x 256 tiles, cut along K where
they do not fill the chip.  Entry by entry against the FP64 product, at the
edges of tiles (256), of the two CTAs' halves (128), of k-steps (64) and of
chunks (320 periods FP32, 1024 else), with and without the optional room for
partials in the workspace."""
import pytest

torch = pytest.importorskip("torch")

pytestmark = pytest.mark.gpu
U = 2.0 ** -24

SHAPES = [(1, 1), (127, 321), (129, 1025), (257, 640), (300, 12345), (1537, 2049), (3300, 1000)]


@pytest.mark.parametrize("shape", SHAPES)
@pytest.mark.parametrize("dt", ["f32", "bf16", "fp8"])
@pytest.mark.parametrize("room", [True, False])
def test_sigma_tiles_and_ranges(shape, dt, room):
    from paper_2604_02917_gb300 import mv

    n, T = shape
    g = torch.Generator(device="cuda")
    g.manual_seed(n + 7 * T)
    A = torch.randn((n, T), generator=g, device="cuda") * 0.01
    scale = None
    if dt == "fp8":
        scale = A.abs().amax(1) / 448
        A = A / scale[:, None]
    kind = {"f32": torch.float32, "bf16": torch.bfloat16, "fp8": torch.float8_e4m3fn}[dt]
    L = torch.zeros((n, mv.padded_ld(T, mv.DTYPES[dt])), device="cuda").to(kind)
    L[:, :T] = A.to(kind)
    W = L[:, :T].to(torch.float64)
    if dt == "fp8":
        L = L.view(torch.uint8)
        W = W * scale.to(torch.float64)[:, None]
    p = mv.make_problem(L, torch.zeros(n, dtype=torch.float64, device="cuda"), 0.0, T, 0.0, dtype=dt, row_scale=scale)
    size = mv.lib().mv_sigma_workspace_size(mv.C.byref(p))
    planes = {"f32": 2, "bf16": 0, "fp8": 1}[dt] * ((n * ((T + 7) // 8 * 8) * 2 + 255) // 256 * 256)
    size = size if room else planes
    ws = torch.empty(size + 256, dtype=torch.uint8, device="cuda")
    ld = (n + 3) // 4 * 4
    S = torch.full((n, ld), 7.0, device="cuda")
    st = mv.lib().mv_sigma_form(mv.C.byref(p), S.data_ptr(), ld, ws.data_ptr() if size else None, size, mv._stream())
    assert st == mv.MV_OK
    assert (S[:, n:] == 7.0).all()                     # the padding is the caller's
    S = S[:, :n]
    assert torch.equal(S, S.T)
    ref, mag = W @ W.T, W.abs() @ W.abs().T
    # one chunk's accumulation (2 ulp per MMA, 64 of them), FP32 sums of chunks and
    # ranges, the dropped split terms (FP32) or the scale products (FP8)
    chunks = -(-(-(-T // 64)) // (5 if dt == "f32" else 16))
    rel = (128 + chunks + 8) * U + (3 * 2.0 ** -18 if dt == "f32" else 0.0)
    assert ((S.double() - ref).abs() <= rel * mag).all()
