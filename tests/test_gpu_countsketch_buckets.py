"""CountSketch over buckets at the edges of the sort's cases: one thread (up to
16 periods), a warp (to 4096), none (above); every sum in ascending order."""
import numpy as np
import pytest

torch = pytest.importorskip("torch")

pytestmark = pytest.mark.gpu


@pytest.mark.parametrize("layout", ["nt", "tn"])
@pytest.mark.parametrize("sizes", [(0, 1, 15, 16, 17, 31, 32, 33, 35), (1023, 1024, 1025, 3, 0), (4095, 4096, 2047), (1500,) * 9,
                                   tuple([3, 16, 17, 200] * 200)])
def test_sums_in_ascending_period_order(layout, sizes):
    from paper_2604_02917_gb300 import mv

    g = np.random.default_rng(len(sizes))
    m, T, n = len(sizes), sum(sizes), 37
    h = np.repeat(np.arange(m), sizes)[g.permutation(T)].astype(np.int32)
    sign = g.choice([-1, 1], T).astype(np.int8)
    A = (g.standard_normal((n, T)) * np.exp(2 * g.standard_normal(T))).astype(np.float32)
    S = A if layout == "nt" else A.T
    L = torch.zeros((S.shape[0], mv.padded_ld(S.shape[1], mv.DTYPES["f32"])), device="cuda")
    L[:, :S.shape[1]] = torch.from_numpy(np.ascontiguousarray(S)).cuda()
    out = mv.countsketch(L, n, T, torch.from_numpy(h).cuda(), torch.from_numpy(sign).cuda(), m, "f32", layout=layout)
    ref = np.zeros((n, m), np.float32)
    for t in range(T):                                     # FP32 additions, one by one
        ref[:, h[t]] += sign[t] * A[:, t]
    np.testing.assert_array_equal(out.cpu().numpy()[:, :m], ref)


def test_a_bucket_above_the_limit_is_refused():
    from paper_2604_02917_gb300 import mv

    T = 4097 + 20
    h = torch.zeros(T, dtype=torch.int32, device="cuda")
    h[4097:] = 1
    L = torch.zeros((8, mv.padded_ld(T, mv.DTYPES["f32"])), device="cuda")
    with pytest.raises(mv.MvError):
        mv.countsketch(L, 8, T, h, torch.ones(T, dtype=torch.int8, device="cuda"), 2)
