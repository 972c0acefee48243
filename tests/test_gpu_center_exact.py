"""mv_center_factor against FP64 arithmetic, entry by entry: the FP32-pair and
integer arithmetic of the kernels must store the rounding of the FP64 value
in every storage type, on rows that leave their fast range too."""
import math

import numpy as np
import pytest

pytestmark = pytest.mark.gpu

# (n, T, extra columns of R): below one warp, ragged tiles (32 assets x 64
# periods, 512 threads x 8 loads), rows of no common alignment.
SHAPES = [(1, 2, 0), (9, 31, 3), (40, 64, 0), (33, 513, 1), (17, 4097, 0), (70, 12345, 5)]


def panel(n, T, seed, finite):
    g = np.random.default_rng(seed)
    R = g.standard_normal((n, T)) * 0.02 + 3e-4
    for i in range(n):
        k = i % 10
        if k == 1:
            R[i, T // 2:] *= 2.0 ** 21                     # the sum's window has to move
        elif k == 2:
            R[i] *= 2.0 ** -70                             # below the FP32 range the pairs rely on
        elif k == 3:
            R[i] *= 2.0 ** 70
        elif k == 4:
            R[i, ::3] = 0.0
        elif k == 5:
            R[i] = 3.7                                     # constant: every entry is its mean
        elif k == 6:
            R[i] = 100.0 + 1e-4 * R[i]                     # mean far above the spread
        elif k == 7:
            R[i] *= np.exp(8 * g.standard_normal(T))       # 40 octaves within a row
        elif k == 8 and not finite:
            R[i, T // 3] = np.nan
        elif k == 9 and not finite:
            R[i, T - 1] = np.inf
    return R.astype(np.float32)


def round_bits(d, bits):
    """FP64 to `bits` significant bits, ties to even."""
    m, e = np.frexp(d)
    return np.ldexp(np.rint(np.ldexp(m, bits)), e - bits)


@pytest.mark.parametrize("shape", SHAPES)
@pytest.mark.parametrize("layout", ["nt", "tn"])
@pytest.mark.parametrize("dt", ["f32", "bf16", "fp8"])
@pytest.mark.parametrize("finite", [True, False])
def test_center_is_the_rounded_fp64_value(shape, layout, dt, finite):
    import torch

    from paper_2604_02917_gb300 import mv

    n, T, pad = shape
    R = panel(n, T, 10 * n + T, finite)
    big = torch.empty((n, T + pad), dtype=torch.float32, device="cuda")
    big[:, :T] = torch.from_numpy(R).cuda()
    L, rs, mu, tr = mv.center_factor(big[:, :T], dt, layout=layout)
    mu = mu.cpu().numpy()
    R64 = R.astype(np.float64)
    # mean: FP64 roundings of the cross-thread sums only (9 shuffle levels and
    # one conversion per thread), so 16 ulp of the mean magnitude bounds it
    for i in range(n):
        if np.isfinite(R64[i]).all():
            exact = math.fsum(R64[i]) / T
            assert abs(mu[i] - exact) <= 2.0 ** -49 * np.abs(R64[i]).mean()
        else:
            assert not np.isfinite(mu[i])
    with np.errstate(invalid="ignore", over="ignore"):
        d = (R64 - mu[:, None]) * (1.0 / math.sqrt(float(T - 1)))
    out = L.cpu()
    out = out[:, :T] if layout == "nt" else out[:T, :n].T
    if layout == "nt":
        assert not L[:, T:].float().abs().any()
    else:
        assert not L[:, n:].float().abs().any()
    d32 = d.astype(np.float32)
    if dt == "f32":
        np.testing.assert_array_equal(out.numpy(), d32)
    elif dt == "bf16":
        np.testing.assert_array_equal(out.to(torch.float64).numpy(), round_bits(d, 8))
    else:
        scale = rs.cpu().numpy()
        with np.errstate(invalid="ignore", divide="ignore"):
            q = torch.from_numpy(d32 * (np.float32(1.0) / scale)[:, None]).clamp(-448, 448).to(torch.float8_e4m3fn)
        ok = np.isfinite(d32)
        np.testing.assert_array_equal(out.contiguous().view(torch.float8_e4m3fn).float().numpy()[ok], q.float().numpy()[ok])
    if finite:
        # pairs: 2^-44 per entry twice, and at most 27 x 64 entries per thread,
        # each adding 2^-48 of the thread's sum
        exact = math.fsum((d * d).ravel())
        assert abs(float(tr) - exact) <= (2.0 ** -42 + 27 * 64 * 2.0 ** -48) * exact
