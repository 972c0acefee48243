"""The latency forms of the two half-products (matrices that do not fill the
machine) against FP64, at the edges of their tiles: rows per split (64),
columns per block, ragged pitches, one and several splits, both layouts."""
import numpy as np
import pytest

pytestmark = pytest.mark.gpu

# (n, T): single rows and columns, one split and its edges, several column
# splits of gemv_n (4096 FP32 / 8192 BF16 / 16384 FP8 columns), many row splits.
SHAPES = [(1, 1), (3, 257), (64, 1000), (65, 1023), (200, 1000), (129, 4097), (40, 16385), (700, 65), (2051, 130), (4100, 33)]


@pytest.mark.parametrize("shape", SHAPES)
@pytest.mark.parametrize("layout", ["nt", "tn"])
@pytest.mark.parametrize("dt", ["f32", "bf16", "fp8"])
def test_gradient_latency_forms(shape, layout, dt):
    import torch

    from paper_2604_02917_gb300 import mv

    n, T = shape
    g = torch.Generator(device="cuda")
    g.manual_seed(n * 100003 + T)
    A = torch.randn((n, T), generator=g, device="cuda") * 0.01
    scale = None
    if dt == "fp8":
        scale = A.abs().amax(1) / 448
        A = A / scale[:, None]
    A = A.T if layout == "tn" else A
    kind = {"f32": torch.float32, "bf16": torch.bfloat16, "fp8": torch.float8_e4m3fn}[dt]
    ld = mv.padded_ld(A.shape[1], mv.DTYPES[dt])
    # the padding holds values that must not count
    L = torch.full((A.shape[0], ld), 3.0, device="cuda").to(kind)
    L[:, :A.shape[1]] = A.to(kind)
    wide = L[:, :A.shape[1]].to(torch.float64)
    wide = wide.T if layout == "tn" else wide
    if dt == "fp8":
        L = L.view(torch.uint8)
        wide = wide * scale.to(torch.float64)[:, None]
    y = torch.rand(n, generator=g, device="cuda", dtype=torch.float64) / n
    z, gr = mv.gradient(L, y, T, 0.25, dt, scale, layout=layout)
    zr = wide.T @ y
    mag_z = wide.abs().T @ y.abs()
    # FP32 input rounding, one rounding per row of a split and per split sum
    assert ((z.double() - zr).abs() <= (n + 8) * 2.0 ** -24 * mag_z + 1e-30).all()
    ref = 2 * wide @ zr + 0.5 * y
    mag = 2 * wide.abs() @ mag_z + 0.5 * y
    # the same for both products (at most 64 + T/64 additions in a column of the transposed form)
    assert ((gr - ref).abs() <= (n + T + 16) * 2.0 ** -24 * mag).all()
    # repeated calls leave the tickets ready and give the same bits
    z2, gr2 = mv.gradient(L, y, T, 0.25, dt, scale, layout=layout)
    assert torch.equal(z, z2) and torch.equal(gr, gr2)
    zn, gn = mv.gradient_noalloc(L, y, T, 0.25, dt, scale, layout)
    assert torch.equal(z, zn) and torch.equal(gr, gn)
