"""The overflow kernels take a 2-bit code as [d > s/2] + [d >= 3s/2] + [d > 5s/2] for d = x - min >= 0 and a bf16
scale s > 0, instead of rounding the quotient d / s (Eq. 1 with the rounding of the quantiser: nearest, ties to even,
clamped at 3).  This checks that identity in IEEE binary32 for EVERY positive finite bf16 scale, at the three
thresholds themselves and at the binary32 neighbours on either side (where the two could differ if they ever
did), and on random d; numpy's float32 division is the correctly rounded one the definition uses."""
import numpy as np
import pytest

pytestmark = pytest.mark.filterwarnings("ignore::RuntimeWarning")  # overflow of 4 * s at the largest scales, filtered out


def _by_division(d, s):
    with np.errstate(over="ignore", invalid="ignore"):
        q = (d / s).astype(np.float32)
    return np.clip(np.rint(q), 0, 3).astype(np.int64)   # np.rint: ties to even


def _by_thresholds(d, s):
    h = np.float32(0.5)
    t1, t2, t3 = h * s, np.float32(1.5) * s, np.float32(2.5) * s
    return (d > t1).astype(np.int64) + (d >= t2).astype(np.int64) + (d > t3).astype(np.int64)


def _all_positive_bf16():
    bits = np.arange(1, 0x7F80, dtype=np.uint32) << 16      # subnormals included, inf and NaN excluded
    return bits.view(np.float32)


def test_threshold_products_are_exact():
    s = _all_positive_bf16().astype(np.float64)
    for c in (0.5, 1.5, 2.5):
        prod = c * s
        ok = np.isfinite(prod.astype(np.float32))
        assert (prod.astype(np.float32).astype(np.float64)[ok] == prod[ok]).all()


def test_codes_by_thresholds_equal_codes_by_rounded_division_near_every_threshold():
    s = _all_positive_bf16()
    s = s[np.isfinite(np.float32(2.5) * s) & np.isfinite(np.float32(4) * s)]
    for c in (0.5, 1.5, 2.5):
        t = np.float32(c) * s
        d = t.copy()
        lo, hi = t.copy(), t.copy()
        cases = [d]
        for _ in range(3):                                   # three binary32 steps to either side
            lo = np.nextafter(lo, np.float32(0))
            hi = np.nextafter(hi, np.float32(np.inf))
            cases += [lo.copy(), hi.copy()]
        for dd in cases:
            assert np.array_equal(_by_thresholds(dd, s), _by_division(dd, s)), c
    # ties go to the even neighbour
    assert _by_thresholds(np.float32([0.5, 1.5, 2.5]), np.float32([1, 1, 1])).tolist() == [0, 2, 2]


def test_codes_by_thresholds_equal_codes_by_rounded_division_on_random_inputs():
    rng = np.random.default_rng(7)
    s = rng.choice(_all_positive_bf16(), size=2_000_000)
    s = s[np.isfinite(np.float32(4) * s)]
    d = (rng.random(len(s)) * 3.2).astype(np.float32) * s    # quotients in [0, 3.2): beyond 3 the clamp applies
    assert np.array_equal(_by_thresholds(d, s), _by_division(d, s))
    # differences of bf16 values, as the kernel forms them (x - min rounded to binary32)
    x = (rng.integers(0, 0x7F80, size=len(s)).astype(np.uint32) << 16).view(np.float32)
    mn = (rng.integers(0, 0x7F80, size=len(s)).astype(np.uint32) << 16).view(np.float32)
    x, mn = np.maximum(x, mn), np.minimum(x, mn)
    with np.errstate(over="ignore", invalid="ignore"):
        d = (x - mn).astype(np.float32)
        sc = ((d / np.float32(3)).astype(np.float32).view(np.uint32) >> 16 << 16).view(np.float32)  # some scale near d/3
    keep = (sc > 0) & np.isfinite(np.float32(4) * sc)
    for dd in (d[keep], (d[keep] * np.float32(0.5)).astype(np.float32), (d[keep] * np.float32(0.83)).astype(np.float32)):
        assert np.array_equal(_by_thresholds(dd, sc[keep]), _by_division(dd, sc[keep]))


# ---- the same comparisons as bf16 thresholds on x itself ----
def _f32(bits16):
    return (np.asarray(bits16, np.int64).astype(np.uint32) << 16).view(np.float32)


def _ordered(s):
    return _f32(np.where(s < 0, 0x8000 - s, s))


def _holds(x, mn, t, strict):
    with np.errstate(invalid="ignore", over="ignore"):
        d = (x - mn).astype(np.float32)
        return d > t if strict else d >= t


def _bisected(mn, t, strict):
    lo, hi = np.full(mn.shape, -0x7F81, np.int64), np.full(mn.shape, 0x7F81, np.int64)
    while (hi - lo > 1).any():
        mid = (lo + hi) >> 1
        up = _holds(_ordered(mid), mn, t, strict)
        hi, lo = np.where(up, mid, hi), np.where(up, lo, mid)
    return _ordered(hi)


def _rounded(mn, t, strict):
    """(threshold, whether the kernel takes it without a search), for finite t"""
    with np.errstate(invalid="ignore", over="ignore"):
        y = (mn + t).astype(np.float32)
        plain = np.abs(y) >= (np.float32(2.0 ** -14) * t).astype(np.float32)
        half = (np.float32(0.5) * (np.nextafter(t, np.float32(np.inf)) - t) if strict
                else np.float32(-0.5) * (t - np.nextafter(t, np.float32(-np.inf)))).astype(np.float32)
        zero = ~plain & (y == 0) & (t >= np.float32(2.0 ** -90))
        y, plain = np.where(zero, half, y), plain | zero
    u = y.view(np.int32).astype(np.int64)
    add = np.where(u >= 0, 0x10000, -1) if strict else np.where(u >= 0, 0xFFFF, 0)
    return _f32(((u + add) & 0xFFFFFFFF) >> 16), plain


def _group_scale(mn, mx):
    with np.errstate(invalid="ignore", over="ignore"):
        q = ((mx - mn).astype(np.float32) / np.float32(3)).astype(np.float32)
    u = q.view(np.uint32).astype(np.uint64)
    r = ((u + 0x7FFF + ((u >> 16) & 1)) >> 16 << 16).astype(np.uint32).view(np.float32)   # bf16, ties to even
    return np.where(np.isfinite(q), r, q)


@pytest.mark.parametrize("kind", ["any", "alike", "symmetric", "small minimum", "subnormal", "lattice"])
def test_bf16_thresholds_taken_without_a_search_are_the_searched_ones(kind):
    rng = np.random.default_rng(len(kind))
    n = 300_000
    bits = rng.integers(0, 0xFF80, size=(2, n))
    if kind == "alike":                                # exponents within a few of one another
        bits = (rng.integers(110, 140, size=n) + rng.integers(-4, 5, size=(2, n))) << 7 | rng.integers(0, 128, size=(2, n)) \
            | rng.integers(0, 2, size=(2, n)) << 15
    elif kind == "symmetric":                          # x near zero decides
        bits[1] = bits[0] ^ 0x8000 ^ rng.integers(0, 3, size=n)
    elif kind == "small minimum":
        bits[0] = (bits[1] & 0x7FFF) - (rng.integers(8, 18, size=n) << 7) + rng.integers(0, 128, size=n) | rng.integers(0, 2, size=n) << 15
        bits[0] = np.clip(bits[0], 0, 0xFF80)
    elif kind == "subnormal":
        bits = rng.integers(0, 0x600, size=(2, n)) | rng.integers(0, 2, size=(2, n)) << 15
    x = _f32(bits)
    if kind == "lattice":                              # min = -k/2 scale and neighbours: the sum with T is zero
        e = np.float32(2.0) ** rng.integers(-20, 20, size=n)
        x = np.stack([-rng.integers(0, 9, size=n) / 2, rng.integers(0, 9, size=n) / 2]).astype(np.float32) * e
    x = x[:, np.isfinite(x).all(0)]
    mn, mx = np.minimum(x[0], x[1]) + np.float32(0), np.maximum(x[0], x[1]) + np.float32(0)
    s = _group_scale(mn, mx)
    keep = (s > 0) & np.isfinite(s)
    mn, mx, s = mn[keep], mx[keep], s[keep]
    with np.errstate(over="ignore"):
        ts = [(np.float32(c) * s).astype(np.float32) for c in (0.5, 1.5, 2.5)]
        base = np.isfinite(ts[2]) & ((mn == 0) | (np.abs(mn) >= (np.float32(2.0 ** -12) * ts[2]).astype(np.float32)))
    rounded = [_rounded(mn, t, strict) for t, strict in zip(ts, (True, False, True))]
    plain = base & rounded[0][1] & rounded[1][1] & rounded[2][1]
    assert plain.mean() > (0.5 if kind in ("alike", "subnormal") else 0.002)
    for (thr, _), t, strict in zip(rounded, ts, (True, False, True)):
        assert np.array_equal(thr[plain], _bisected(mn[plain], t[plain], strict))
