"""The integer-pipe conversions between FP64 and float pairs (csrc/f64_bits.cuh),
emulated step by step in numpy: equal to the floating-point expressions they
stand for (round to nearest even at every step), over random values, exact
ties, carries into the next binade, powers of two and the edges of their ranges."""
import numpy as np


def split(x):
    """split_f64: (h, l, took the fast path)."""
    b = np.asarray(x, np.float64).view(np.uint64)
    hi, lo = (b >> np.uint64(32)).astype(np.int64), (b & np.uint64(0xFFFFFFFF)).astype(np.int64)
    ex = (hi >> 20) & 0x7FF
    fast = (ex >= 963) & (ex < 963 + 180)
    f = ((ex - 896) << 23) | ((hi & 0xFFFFF) << 3) | (lo >> 29)
    rem = lo & 0x1FFFFFFF
    up = (rem + (f & 1) > 0x10000000).astype(np.int64)
    f = f + up
    r = rem - (up << 29)
    s = hi & 0x80000000
    h = ((f | s) & 0xFFFFFFFF).astype(np.uint32).view(np.float32)
    with np.errstate(all="ignore"):
        l = np.where(s != 0, -r, r).astype(np.float32) * np.ldexp(1.0, np.clip(ex - 1075, -126, 127)).astype(np.float32)
    return h, l.astype(np.float32), fast


def join(h, l):
    """join_f64: (sum, took the fast path)."""
    h, l = np.asarray(h, np.float32), np.asarray(l, np.float32)
    hb = h.view(np.uint32).astype(np.int64)
    eh, fh = (hb >> 23) & 0xFF, hb & 0x7FFFFF
    with np.errstate(all="ignore"):
        L = (l * np.ldexp(np.float32(1), np.clip(179 - eh, -126, 127)).astype(np.float32)).astype(np.float32)
        inward = ((hb ^ L.view(np.uint32).astype(np.int64)) & 0x80000000) != 0
        fast = (eh >= 52) & (eh < 247) & (np.abs(L) <= 268435456.0) & ~(inward & (fh == 0))
        d = np.where(fast, np.rint(np.abs(L)), 0).astype(np.int64)
    m = (fh << 29) + np.where(inward, -d, d)
    bits = ((hb & 0x80000000).astype(np.uint64) << np.uint64(32)) | (((eh + 896) << 52) + m).astype(np.uint64)
    return bits.view(np.float64), fast


def _values():
    rng = np.random.default_rng(11)
    x = np.ldexp(rng.uniform(1.0, 2.0, 400000), rng.integers(-64, 124, 400000)) * rng.choice([-1.0, 1.0], 400000)
    m = rng.integers(0, 2 ** 23, 20000).astype(np.float64)
    ties = np.ldexp(2.0 ** 23 + m + 0.5, rng.integers(-80, 90, 20000))          # halfway between two floats
    near = np.concatenate([np.nextafter(ties, 0), np.nextafter(ties, np.inf)])
    carry = np.ldexp(2.0 - rng.integers(0, 4, 2000) * 2.0 ** -52, rng.integers(-55, 110, 2000))
    pow2 = np.ldexp(1.0, np.arange(-59, 119))
    return np.concatenate([x, ties, -ties, near, carry, -carry, pow2, -pow2])


def test_split_equals_the_rounded_pair():
    x = _values()
    h, l, fast = split(x)
    rh = x.astype(np.float32)
    rl = (x - rh.astype(np.float64)).astype(np.float32)
    assert fast.mean() > 0.9
    np.testing.assert_array_equal(h[fast].view(np.uint32), rh[fast].view(np.uint32))
    np.testing.assert_array_equal(l[fast].view(np.uint32), rl[fast].view(np.uint32))


def test_join_equals_the_sum():
    rng = np.random.default_rng(12)
    x = _values()
    h = x.astype(np.float32)
    l = (x - h.astype(np.float64)).astype(np.float32)
    # pairs with lower bits below the sum's last place, ties at it, zero and opposite low parts
    e = np.frexp(np.abs(h))[1]
    l2 = (rng.uniform(-0.5, 0.5, h.size) * np.ldexp(1.0, e - 24)).astype(np.float32)
    l3 = ((rng.integers(-2 ** 20, 2 ** 20, h.size) + 0.5) * np.ldexp(1.0, e - 53)).astype(np.float32)
    for low in (l, l2, l3, np.zeros_like(h), -l, (l2 * np.float32(2.0 ** -30)).astype(np.float32)):
        s, fast = join(h, low)
        ref = h.astype(np.float64) + low.astype(np.float64)
        assert fast.mean() > 0.8
        np.testing.assert_array_equal(s[fast].view(np.uint64), ref[fast].view(np.uint64))
