"""Rules of the loop kernel that give a costlier form's answer by other
arithmetic, checked on the host against that form: the kernel's own functions
(kp_arith.cuh, kp_layout.h), compiled into tests/host/kp_arith_harness.cu."""
import ctypes as C
import os
import shutil
import subprocess

import numpy as np
import pytest

ROOT = os.path.dirname(os.path.dirname(os.path.abspath(__file__)))
SRC = os.path.join(ROOT, "tests", "host", "kp_arith_harness.cu")
OUT = os.path.join(ROOT, "tests", "host", "_build", "libkparith.so")
CSRC = os.path.join(ROOT, "paper_2409_06807_gb300", "csrc")


@pytest.fixture(scope="module")
def H():
    nvcc = shutil.which("nvcc") or "/usr/local/cuda/bin/nvcc"
    if not os.path.exists(nvcc):
        pytest.skip("nvcc is needed to build the host harness")
    deps = [SRC] + [os.path.join(CSRC, f) for f in ("kp_arith.cuh", "kp_layout.h")]
    if not os.path.exists(OUT) or any(os.path.getmtime(p) > os.path.getmtime(OUT) for p in deps):
        os.makedirs(os.path.dirname(OUT), exist_ok=True)
        tmp = OUT + f".tmp{os.getpid()}"
        # no products contracted into sums, and rounding modes respected
        subprocess.run([nvcc, "-gencode", "arch=compute_103a,code=sm_103a", "-O2", "-std=c++17",
                        "-Xcompiler", "-fPIC,-ffp-contract=off,-frounding-math", "-shared",
                        "-o", tmp, SRC, "-cudart", "static"], check=True)
        os.replace(tmp, OUT)
    L = C.CDLL(OUT)

    def arr(t):
        return np.ctypeslib.ndpointer(t, flags="C_CONTIGUOUS")

    i32, u32, u64, f32, f64, u8 = (arr(t) for t in (np.int32, np.uint32, np.uint64, np.float32,
                                                    np.float64, np.uint8))
    L.kpt_key_quot.argtypes = [C.c_int, i32, C.c_int, i32]
    L.kpt_bias.argtypes = [C.c_int] * 3
    L.kpt_within.argtypes = [f32, C.c_int, C.c_int, u8]
    L.kpt_threshold_of.argtypes = [f64, C.c_int, u64]
    L.kpt_thresholds.argtypes = [f64, C.c_int, C.c_double, C.c_double, u64, u64]
    L.kpt_draws.argtypes = [u32, f64, C.c_int, C.c_double, C.c_double, u8, u8]
    return L


def test_key_division_is_exact(H):
    """Every lambda, at the keys around every kind of edge of [0, 2^30)."""
    rng = np.random.default_rng(0)
    for lam in range(1, 1025):
        top = (1 << 30) // lam
        q = np.unique(np.concatenate([np.arange(0, 64), rng.integers(0, top, 200),
                                      np.arange(max(0, top - 64), top)]))
        q = q[q < top]
        for off in {0, min(1, lam - 1), lam - 1}:
            key = np.ascontiguousarray(q * lam + off, dtype=np.int32)
            got = np.empty_like(key)
            H.kpt_key_quot(lam, key, len(key), got)
            assert key.max() < 1 << 30 and np.array_equal(got, key // lam)


@pytest.mark.parametrize("g", [(16, 16, 16), (64, 64, 1), (1, 64, 64), (4, 32, 32), (1, 1, 1)])
def test_biased_cell_words_add_up_to_the_cell(H, g):
    bias = H.kpt_bias(*g) & 0xFFFFFFFF
    for x in {0, g[0] - 1}:
        for y in {0, g[1] - 1}:
            for z in {0, g[2] - 1}:
                w = [int((np.float32(8388608.0) + np.float32(v)).view(np.uint32)) for v in (x, y, z)]
                got = (w[0] + g[0] * w[1] + g[0] * g[1] * w[2] - bias) & 0xFFFFFFFF
                assert got == x + g[0] * (y + g[1] * z)


def test_clearance_comparison_in_integers(H):
    """d <= 1 + q / 16 for every byte q, at distances on and next to the edge,
    far below and far above it (the clearance is capped at 4 cells); byte 0 says
    that nothing is known."""
    for q in range(0, 64):
        edge = np.float32(1.0 + q / 16.0)
        d = np.array([0.0, 1e-30, 0.5, 1.0, edge, np.nextafter(edge, np.float32(0)),
                      np.nextafter(edge, np.float32(9)), 300.0, 1e9, np.inf], np.float32)
        got = np.empty(len(d), np.uint8)
        H.kpt_within(d, len(d), q, got)
        want = (d.astype(np.float64) <= 1.0 + q / 16.0) & (q > 0)
        assert np.array_equal(got.astype(bool), want), q


def thresholds_of(H, p):
    p = np.ascontiguousarray(p, np.float64)
    out = np.empty(len(p), np.uint64)
    H.kpt_threshold_of(p, len(p), out)
    return out


def test_threshold_from_the_bits(H):
    """floor(min(p, 1) 2^32): every binary exponent, the neighbours of whole
    thresholds, 1 and above, infinity and NaN (neither compares below 1)."""
    rng = np.random.default_rng(1)
    p = [2.0 ** e * m for e in range(-80, 3) for m in (1.0, 1.0 + 2.0**-52, 1.5, 2.0 - 2.0**-52)]
    for k in [1, 2, 3, 2**31, 2**32 - 1, 2**32, *rng.integers(1, 2**32, 200).tolist()]:
        p += [k / 2.0**32, np.nextafter(k / 2.0**32, 0.0), np.nextafter(k / 2.0**32, 9.0)]
    p += [5e-324, 1e300]
    want = [int(np.floor(min(v, 1.0) * 2.0**32)) for v in p]
    assert thresholds_of(H, p).tolist() == want
    assert thresholds_of(H, [np.inf, np.nan, -np.nan]).tolist() == [1 << 32] * 3


def exact_threshold(H, score, total, eps):
    """Eq. 5 with the division, in FP64 (score -1: outside R_avail)."""
    with np.errstate(all="ignore"):
        p = score / total + eps if total > 0 else np.full(len(score), eps)
    return np.where(score == -1.0, np.uint64(1 << 32), thresholds_of(H, p))


EPS = [1e-300, 1e-12, 1e-4, 0.01, 0.5, 0.9]


def draws(H, w, score, total, eps):
    w, score = np.ascontiguousarray(w, np.uint32), np.ascontiguousarray(score, np.float64)
    out, decided = np.empty(len(w), np.uint8), np.empty(len(w), np.uint8)
    H.kpt_draws(w, score, len(w), total, eps, out, decided)
    return out.astype(bool), decided.astype(bool)


def test_acceptance_without_the_division(H):
    """Scores over 40 binary orders, regions without one among them, the draws
    on, next to and around the threshold, eps from 1e-300 to 0.9: what is decided
    without the division is decided as with it, the draws right at a threshold
    take the threshold itself, and few random draws need it."""
    rng = np.random.default_rng(2)
    undecided = total_draws = at_edge = 0
    for _ in range(400):
        n = int(rng.integers(1, 50))
        s = np.exp2(rng.uniform(-40, 0, n) - rng.integers(0, 600)) * (rng.random(n) > 0.1)
        total, eps = float(s.sum()), float(rng.choice(EPS))
        if not total > 0:
            continue
        s[rng.random(n) < 0.05] = -1.0
        want = exact_threshold(H, s, total, eps)
        fast, slow = np.empty(n, np.uint64), np.empty(n, np.uint64)
        assert H.kpt_thresholds(s, n, total, eps, fast, slow) == 1
        assert np.array_equal(fast, want) and np.array_equal(slow, want)
        around = want[:, None].astype(np.int64) + np.arange(-3, 4)
        w = np.concatenate([around, np.broadcast_to([0, 1, 2**32 - 1], (n, 3)),
                            rng.integers(0, 2**32, (n, 8))], 1)
        ok = (w >= 0) & (w < 2**32)
        sc, th = np.broadcast_to(s[:, None], w.shape)[ok], np.broadcast_to(want[:, None], w.shape)[ok]
        got, decided = draws(H, w[ok], sc, total, eps)
        assert np.array_equal(got, w[ok].astype(np.uint64) < th)
        rand = np.zeros(w.shape, bool)
        rand[:, -8:] = True
        undecided += int((~decided & rand[ok]).sum())
        total_draws += int(rand[ok].sum())
        at_edge += int((~decided & ~rand[ok]).sum())
    assert undecided < 0.01 * total_draws and at_edge > 10000


def test_thresholds_on_their_edge(H):
    """Scores that are a whole number of 2^-32 parts of the sum, and their
    neighbours: the quotient is on a threshold's edge or next to it, and the
    product with 1 / sum falls on either side."""
    rng = np.random.default_rng(4)
    sides = set()
    for total in (2 * rng.integers(1, 1 << 19, 200) + 1).astype(np.float64):
        k = rng.integers(1, 1 << 32, 50).astype(np.float64)
        s = k * total * 2.0**-32  # exact: below 2^53 before the power of two
        assert np.array_equal(exact_threshold(H, s, total, 1e-300), k.astype(np.uint64))
        sides |= set(np.sign(s * (1.0 / total) - k * 2.0**-32).tolist())
        s = np.concatenate([s, np.nextafter(s, 0.0), np.nextafter(s, 2 * s)])
        want = exact_threshold(H, s, total, 1e-300)
        fast, slow = np.empty(len(s), np.uint64), np.empty(len(s), np.uint64)
        H.kpt_thresholds(s, len(s), total, 1e-300, fast, slow)
        assert np.array_equal(fast, want) and np.array_equal(slow, want)
    assert sides == {-1.0, 0.0, 1.0}


@pytest.mark.parametrize("total", [0.0, 5e-324, 1e-300, 2.0**-901, 2.0**901, 1e300, np.inf, np.nan])
def test_sums_without_an_inverse(H, total):
    """A sum that is not a number between 2^-900 and 2^900 has no inverse: every
    threshold is taken with the division and every draw from the threshold, with
    scores of the sum's size and below, none, infinite and no numbers (whose sign
    bit must not make them a region without a score)."""
    rng = np.random.default_rng(3)
    base = total if np.isfinite(total) and total > 0 else 1.0
    s = np.array([0.0, base, base / 3, base * 1e-5, -1.0, np.inf, np.nan, -np.nan], np.float64)
    s = s[np.array([True, True, True, True, True] + [not np.isfinite(total)] * 3)]
    for eps in EPS:
        want = exact_threshold(H, s, total, eps)
        fast, slow = np.empty(len(s), np.uint64), np.empty(len(s), np.uint64)
        assert H.kpt_thresholds(s, len(s), total, eps, fast, slow) == 0
        assert np.array_equal(fast, want) and np.array_equal(slow, want)
        w = np.concatenate([want[:, None].astype(np.int64) + np.arange(-2, 3),
                            rng.integers(0, 2**32, (len(s), 6))], 1)
        ok = (w >= 0) & (w < 2**32)
        sc = np.broadcast_to(s[:, None], w.shape)[ok]
        got, decided = draws(H, w[ok], sc, total, eps)
        assert np.array_equal(got, w[ok].astype(np.uint64) < np.broadcast_to(want[:, None], w.shape)[ok])
        assert not decided[sc != -1.0].any()
