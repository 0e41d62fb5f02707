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
