"""mv_center_factor: an infinity or a NaN decides its row's mean whatever the
magnitude of the values beside it."""
import numpy as np
import pytest

pytestmark = pytest.mark.gpu


# (T, dtype, layout): a row in one thread's reach, and rows that 512 and 128 threads share
@pytest.mark.parametrize("T", [4, 4099, 9001])
@pytest.mark.parametrize("layout", ["nt", "tn"])
@pytest.mark.parametrize("dt", ["f32", "bf16", "fp8"])
@pytest.mark.parametrize("rows", [16, 1300])
def test_mean_of_rows_with_nonfinite_values(T, layout, dt, rows):
    import torch

    from paper_2604_02917_gb300 import mv

    big = [2e30, 2e36, 1.7e38, 3e38, -2e36, 1.0]          # below, at and above 2^120, and an ordinary row
    tails = [(), (np.inf,), (-np.inf,), (np.nan,), (np.inf, -np.inf), (np.nan, np.inf)]
    R = np.full((rows, T), 1.0, np.float32)
    for i in range(rows):
        b, tail = big[i % len(big)], tails[i // len(big) % len(tails)]
        R[i] = np.float32(b) * np.where(np.arange(T) % 2, 1.0, 0.5).astype(np.float32)
        # behind finite values of the same threads: 8 loads of 512 threads precede them where the row is long enough
        for k, v in enumerate(tail):
            R[i, T - 1 - k] = v
    mu = mv.center_factor(torch.from_numpy(R).cuda(), dt, layout=layout)[2].cpu().numpy()
    with np.errstate(invalid="ignore"):
        ref = R.astype(np.float64).sum(1) / T
    np.testing.assert_array_equal(np.isnan(mu), np.isnan(ref))
    np.testing.assert_array_equal(np.isinf(mu), np.isinf(ref))
    np.testing.assert_array_equal(np.sign(mu[np.isinf(ref)]), np.sign(ref[np.isinf(ref)]))
    ok = np.isfinite(ref)
    # 16 ulp of the mean magnitude: conversions per thread and the sums over threads
    assert (np.abs(mu[ok] - ref[ok]) <= 2.0 ** -49 * np.abs(R[ok].astype(np.float64)).mean(1)).all()
