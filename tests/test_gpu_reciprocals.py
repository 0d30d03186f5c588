"""The kernels' own 1 / sqrt(v) and 1 / v (an FP32 seed and one step of Householder's third-order iteration) over the whole
exponent range: random significands, those just above 1 and just below 2, the limits of the two ranges, zero, subnormals,
negative values, infinities and NaN.

Bounds. The seeds are off by at most 2^-21 (the value cut to 24 bits, then two units of FP32), the iteration leaves
their cube, 2^-63, and rounding: for 1 / v that of one fma (half an ulp), for 1 / sqrt(v) also that of v y in the residual
(half of 2^-53): within one ulp (2^-52 relative) and one and a half of the exact values. Outside of the ranges the
library's bits."""
import numpy as np
import pytest

pytestmark = pytest.mark.gpu


def test_reciprocals_against_the_library():
    torch = pytest.importorskip("torch")
    if not torch.cuda.is_available():
        pytest.skip("no CUDA device")
    import paper_2201_05529_gb300 as pkg
    pkg.build()
    capi = pkg.load()
    capi.use_torch_allocator()
    rng = np.random.default_rng(11)
    mant = rng.integers(0, 1 << 52, size=(400, 2046), dtype=np.uint64)
    edge = np.array([0, 1, 2, (1 << 23) - 1, 1 << 28, (1 << 29) - 1, 1 << 29, (1 << 51) - 1, 1 << 51, (1 << 52) - 2,
                     (1 << 52) - 1], dtype=np.uint64)
    mant = np.concatenate([mant, np.repeat(edge[:, None], 2046, axis=1)])
    bits = mant | (np.arange(1, 2047, dtype=np.uint64) << np.uint64(52))[None, :]
    normal = bits.reshape(-1).view(np.float64)
    tiny = 5e-324 * 2.0 ** np.arange(0, 52)
    other = np.concatenate([tiny, np.nextafter(2.0 ** -1022, 0) * np.ones(1), [0.0, -0.0, np.inf, -np.inf, np.nan],
                            -normal[:5000], -tiny])
    v = np.concatenate([normal, other])
    out = torch.zeros((4, v.size), dtype=torch.float64, device="cuda")
    capi.selftest_reciprocals(torch.from_numpy(v).cuda(), out)
    rs, rs0, rc, rc0 = out.cpu().numpy()
    n = normal.size
    x = normal.astype(np.longdouble)
    # relative errors, of quantities scaled into the normal range where 1 / v is subnormal (v above 2^1022)
    assert np.abs(rs[:n].astype(np.longdouble) * np.sqrt(x) - 1).max() <= 1.5 * 2.0 ** -52
    ok = normal < 2.0 ** 1022
    assert np.abs(rc[:n][ok].astype(np.longdouble) * x[ok] - 1).max() <= 2.0 ** -52
    same = lambda a, b: np.array_equal(a.view(np.int64)[~np.isnan(a)], b.view(np.int64)[~np.isnan(b)]) and \
        np.array_equal(np.isnan(a), np.isnan(b))
    assert same(rs[n:], rs0[n:]) and same(rc[n:], rc0[n:])
    hi = normal.view(np.uint64) >> np.uint64(32)
    out_of_range = (hi < 0x00300000) | (hi >= 0x7fd00000)
    assert out_of_range.any() and same(rc[:n][out_of_range], rc0[:n][out_of_range])
