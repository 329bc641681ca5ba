"""The integer recipes that keep conversions off the FP64 pipe, restated in
numpy and compared with numpy's own conversions: FP64 -> FP32 to nearest even
(the downshifted step's coefficients) and the truncated FP32 head of an FP64
value (the FP64 form's inside test and exit-face order)."""
import numpy as np
import pytest


def _values(kind):
    rng = np.random.default_rng(12)
    if kind == "wide":      # signs, magnitudes across the FP32 range
        return np.concatenate([s * rng.random(20000) * 2.0 ** rng.uniform(-126, 126, 20000) for s in (1, -1)])
    if kind == "ties":      # halfway between floats, and one FP64 ulp to either side
        f = np.abs(rng.standard_normal(20000)).astype(np.float32)
        mid = (f.astype(np.float64) + np.nextafter(f, np.float32(np.inf)).astype(np.float64)) / 2
        return np.concatenate([mid, np.nextafter(mid, 0), np.nextafter(mid, 9.0), f.astype(np.float64)])
    return np.array([2.0 ** -126, 2.0 ** 126, 1 - 2.0 ** -25, 1 - 2.0 ** -24, 2 - 2.0 ** -25, 2.0 ** 127 * (1 - 2.0 ** -30)])


def _words(r):
    u = r.view(np.uint64)
    return (u >> np.uint64(32)).astype(np.uint32), (u & np.uint64(0xffffffff)).astype(np.uint32)


@pytest.mark.parametrize("kind", ["wide", "ties", "edges"])
def test_round32(kind):
    r = _values(kind)
    hi, lo = _words(r)
    e = (hi >> 20) & 0x7ff
    ok = (e >= 897) & (e < 1150)     # the recipe's range; the kernel takes the hardware conversion elsewhere
    m = ((e - 896) << 23) | ((hi & 0xfffff) << 3) | (lo >> 29)
    rest = lo & 0x1fffffff
    up = (rest > 0x10000000) | ((rest == 0x10000000) & ((m & 1) == 1))
    f = ((hi & 0x80000000) | (m + up.astype(np.uint32))).astype(np.uint32).view(np.float32)
    assert ok.any() and np.array_equal(f[ok], r[ok].astype(np.float32))


@pytest.mark.parametrize("kind", ["wide", "ties", "edges"])
def test_trunc32(kind):
    r = _values(kind)
    hi, lo = _words(r)
    e = (hi >> 20) & 0x7ff
    ok = (e >= 897) & (e <= 1150)
    f = ((hi & 0x80000000) | ((e - 896) << 23) | ((hi & 0xfffff) << 3) | (lo >> 29)).astype(np.uint32).view(np.float32)
    f, r = f[ok].astype(np.float64), r[ok]
    assert np.all(np.abs(f) <= np.abs(r)) and np.all(np.abs(r) - np.abs(f) <= np.abs(r) * 2.0 ** -23)
    assert np.array_equal(np.sign(f), np.sign(r))
