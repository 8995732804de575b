"""The rule the refinement residual uses to form fl32(r * inv), inv a power of
two, on the bit fields: over the exponent range it accepts the float equals the
FP64 product narrowed once (numpy rounds to nearest even), ties, near-ties and
all-ones mantissas included, and it accepts no subnormal, infinite or NaN r."""
import numpy as np
import pytest


def narrow(r, k):
    bias = k - 896
    b = r.view(np.uint64)
    hi, lo = (b >> np.uint64(32)).astype(np.uint32), b.astype(np.uint32)
    ef = ((hi >> 20) & 0x7ff).astype(np.int64) + bias
    ok = (ef >= 1) & (ef <= 253) & (-1793 <= bias <= 0)
    up = (lo + np.uint32(0x0fffffff) + ((lo >> 29) & 1)).astype(np.uint32)
    m = ((np.where(ok, ef, 0).astype(np.uint32) << 20) | (hi & 0xfffff)) + (up < lo).astype(np.uint32)
    bits = (hi & np.uint32(0x80000000)) | ((m << np.uint32(3)) | (up >> np.uint32(29))).astype(np.uint32)
    return ok, bits.view(np.float32)


@pytest.mark.parametrize("k", [-1022, -897, -300, -20, 0, 5, 300, 896, 1000])
def test_narrowed_bits_equal_the_narrowed_product(k):
    rng = np.random.default_rng(k + 2000)
    n = 400_000
    e = np.clip(rng.integers(1023 - k - 160, 1023 - k + 160, n), 0, 2047).astype(np.uint64)
    m = rng.integers(0, 1 << 52, n, dtype=np.uint64)
    kind = rng.integers(0, 4, n)
    ones = np.uint64((1 << 52) - (1 << 29))
    tie = np.uint64(1 << 28)
    m = np.where(kind == 1, (m & ones) | tie, np.where(kind == 2, m | ones, np.where(kind == 3, ones | tie, m)))
    r = ((rng.integers(0, 2, n).astype(np.uint64) << np.uint64(63)) | (e << np.uint64(52)) | m).view(np.float64)
    ok, f = narrow(r, k)
    assert ok.any() == (-897 <= k <= 896)
    if -300 <= k <= 300:
        assert ok.mean() > 0.5
    assert np.isfinite(r[ok]).all() and (np.abs(r[ok]) >= np.finfo(np.float64).tiny).all()
    with np.errstate(all="ignore"):
        want = np.ldexp(r, k).astype(np.float32)
    assert np.array_equal(f[ok].view(np.uint32), want[ok].view(np.uint32))
