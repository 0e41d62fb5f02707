"""Rules of the propagate phase that select a cheaper form of the same
arithmetic, checked on the host: the multiplication that divides a sample key
by lambda (KeyDiv), the cell index from biased cell words (bp_bias_of) and the
clearance comparison in integers (hull_clear)."""
import numpy as np
import pytest


def key_mul(lam):
    s = lam.bit_length() - 1
    a, b = divmod(0x80000000, lam)
    c, d = divmod(b << s, lam)
    return s, (a << s) + c + (1 if d else 0)


def test_key_division_is_exact():
    """Every lambda, at the keys around every kind of edge of [0, 2^28]."""
    rng = np.random.default_rng(0)
    for lam in range(1, 1025):
        s, mul = key_mul(lam)
        assert mul == -(-(1 << (31 + s)) // lam) and mul <= 1 << 31
        top = (1 << 28) // lam
        q = np.unique(np.concatenate([np.arange(0, 64), rng.integers(0, top + 1, 200),
                                      np.arange(max(0, top - 64), top + 1)])).astype(np.uint64)
        for off in (0, 1, lam - 1):
            key = q * np.uint64(lam) + np.uint64(off)
            assert np.array_equal((key * np.uint64(2) * np.uint64(mul) >> np.uint64(32)) >> np.uint64(s),
                                  key // np.uint64(lam))


@pytest.mark.parametrize("g", [(16, 16, 16), (64, 64, 1), (1, 64, 64), (4, 32, 32), (1, 1, 1)])
def test_biased_cell_words_add_up_to_the_cell(g):
    bias = 0x4B000000 * (1 + g[0] + g[0] * g[1])
    for x in {0, g[0] - 1}:
        for y in {0, g[1] - 1}:
            for z in {0, g[2] - 1}:
                w = [int((np.float32(8388608.0) + np.float32(v)).view(np.uint32)) for v in (x, y, z)]
                got = (w[0] + g[0] * w[1] + g[0] * g[1] * w[2] - bias) & 0xFFFFFFFF
                assert got == x + g[0] * (y + g[1] * z)


def test_clearance_comparison_in_integers():
    """16 d - 16 rounded up against q decides d <= 1 + q / 16, for every byte q
    and distances on and next to the decision's edge (at most 4 cells of
    clearance, so the sums are exact in FP64 here)."""
    for q in range(1, 65):
        edge = np.float32(1.0 + q / 16.0)
        for d in (np.float32(0.0), np.float32(0.5), np.float32(1.0), edge,
                  np.nextafter(edge, np.float32(0)), np.nextafter(edge, np.float32(9)), np.float32(300.0)):
            up = int(np.ceil(float(d) * 16.0 - 16.0))  # fused, rounded up to the integers' spacing
            assert (up <= q) == (float(d) <= 1.0 + q / 16.0)


def threshold_of(p):
    bits = int(np.float64(p).view(np.uint64))
    e = (bits >> 52) - 1023
    if e >= 0:
        return 1 << 32
    mant = (bits & ((1 << 52) - 1)) | (1 << 52)
    return mant >> (20 - e) if 20 - e < 64 else 0


def test_threshold_from_the_bits():
    """floor(min(p, 1) 2^32): every binary exponent, the neighbours of whole
    thresholds, 1 and above, infinity and NaN (neither compares below 1)."""
    rng = np.random.default_rng(1)
    p = [2.0 ** e * m for e in range(-80, 3) for m in (1.0, 1.0 + 2.0**-52, 1.5, 2.0 - 2.0**-52)]
    for k in [1, 2, 3, 2**31, 2**32 - 1, 2**32, *rng.integers(1, 2**32, 200).tolist()]:
        p += [k / 2.0**32, np.nextafter(k / 2.0**32, 0.0), np.nextafter(k / 2.0**32, 9.0)]
    p += [5e-324, 1e300]
    for v in p:
        assert threshold_of(v) == int(np.floor(min(v, 1.0) * 2.0**32)), v
    for v in (np.inf, np.nan, -np.nan):
        assert threshold_of(v) == 1 << 32


def exact_threshold(score, total, eps):
    return threshold_of(score / total + eps if total > 0 else eps)


def fast_threshold(score, inv, eps):
    """accept_threshold's answer without the division, None where it divides."""
    near = int(np.float64(np.longdouble(score) * np.longdouble(inv) + np.longdouble(eps)).view(np.int64))
    lo, hi = (threshold_of(np.int64(near + d).view(np.float64)) for d in (-16, 16))
    return lo if lo == hi else None


def fast_draw(w, score, inv, eps):
    """draw_accepted's answer in FP32, None where it takes the threshold."""
    f = np.float32
    m, e = np.frexp(score)
    im, ie = np.frexp(inv)
    e = int(e) - 1 + int(ie) - 1 if score > 0 else -2000
    m = f(np.floor(m * 2.0**24) / 2.0**23) if score > 0 else f(1.0)
    scale = f(0.0) if e < -126 else f(2.0) ** f(e)
    r = f(np.float64(f(m * f(im * 2.0))) * np.float64(scale) + np.float64(f(eps)))
    t, w1 = f(r * f(4294967296.0)), f(f(w) + f(1.0))
    if abs(f(t - w1)) > f(max(t, w1) * f(2.0**-18)):
        return bool(w1 < t)
    return None


def test_acceptance_without_the_division():
    """Scores over 40 binary orders, the draws on, next to and around the
    threshold, eps from 1e-300 to 0.9: what is decided without the division is
    decided as with it, and few random draws need it."""
    rng = np.random.default_rng(2)
    undecided = draws = 0
    for _ in range(300):
        n = int(rng.integers(1, 50))
        s = np.exp2(rng.uniform(-40, 0, n) - rng.integers(0, 600)) * (rng.random(n) > 0.1)
        total, eps = s.sum(), float(rng.choice([1e-300, 1e-12, 1e-4, 0.01, 0.5, 0.9]))
        if not total > 0:
            continue
        inv = 1.0 / total
        for score in s[:6]:
            thr = exact_threshold(score, total, eps)
            fast = fast_threshold(score, inv, eps)
            assert fast is None or fast == thr
            for w in {0, 1, thr - 2, thr - 1, thr, thr + 1, 2**32 - 1, *rng.integers(0, 2**32, 4).tolist()}:
                if 0 <= w < 2**32:
                    d = fast_draw(w, score, inv, eps)
                    assert d is None or d == (w < thr)
            for w in rng.integers(0, 2**32, 4).tolist():
                draws += 1
                undecided += fast_draw(w, score, inv, eps) is None
    assert undecided < 0.01 * draws
