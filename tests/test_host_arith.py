"""Arithmetic identities the kernels rely on, checked on the CPU in IEEE FP32 (numpy's float32
operations are correctly rounded, as the device's are with -prec-div / -prec-sqrt)."""
import numpy as np


def test_reciprocal_quotient_is_exact_below_2_16():
    """The voxel enumeration of the candidate kernels takes floor(i / n) as the integer part
    of (i + 0.5) * fl(1/n) in FP32, for ranges of at most 2^16 voxels.  The rounding error,
    at most (i / n) 2^-23, stays below the 0.5 / n margin.  Checked for every n up to 4096 and
    a spread of larger n, against every i < 2^16."""
    i = np.arange(65536, dtype=np.int64)
    fi = i.astype(np.float32) + np.float32(0.5)
    ns = list(range(1, 4097)) + list(range(4097, 65537, 97)) + [65535, 65536]
    for n in ns:
        inv = np.float32(1.0) / np.float32(n)
        q = (fi * inv).astype(np.int64)
        assert np.array_equal(q, i // n), n


def test_sign_of_rounded_difference_decides_the_order():
    """FP32 subtraction of finite values rounds to zero only for equal operands, so the sign
    of fl(a - b) is the sign of a - b (the per-row set and open tests of the capsule steps are
    comparisons against a budget; this is the identity their derivation uses)."""
    rng = np.random.default_rng(7)
    a = rng.standard_normal(200000).astype(np.float32) * np.float32(3.0)
    b = (a + rng.standard_normal(200000).astype(np.float32) * np.float32(1e-6)).astype(np.float32)
    d = a - b
    assert np.array_equal(d > 0, a > b) and np.array_equal(d < 0, a < b) and np.array_equal(d == 0, a == b)


def _round_24(n):
    """Integers rounded to 24 significant bits, ties to even."""
    mag = np.abs(n)
    bits = np.zeros_like(mag)
    for s in (32, 16, 8, 4, 2, 1):
        up = (mag >> bits) >> s > 0
        bits += np.where(up, s, 0)
    drop = np.maximum(bits + 1 - 24, 0)
    half = (1 << drop) >> 1
    low = mag & ((1 << drop) - 1)
    q = mag >> drop
    q += (low > half) | ((low == half) & (drop > 0) & (q & 1 == 1))
    return np.sign(n) * (q << drop)


def _markstein_quotient(A, B):
    """fl(q + fl(a - q b) r), q = fl(a r), r = fl(1 / b), for 24-bit integers, as (integer, units): the FP32
    operations in integers."""
    R = (2 ** 48 // B + 1) // 2                       # 1 / B = R 2^-47 (never a tie; B is no power of two)
    P = A * R
    s = np.where(P >= 1 << 47, 24, 23)
    Q = _round_24(P) >> s
    N = _round_24((A << (47 - s)) - Q * B)
    F = N * R                                         # result: Q + F / 2^47
    f = F >> 47
    low = F - (f << 47)
    up = (low > 1 << 46) | ((low == 1 << 46) & ((Q + f) & 1 == 1))
    return Q + f + up, s


def test_corrected_quotient_is_correctly_rounded():
    """vx_div corrects a r once by the remainder.  r carries half an ulp of 1 / b, so the estimate is within
    1.5 ulp and the sum before its rounding within 2.25 * 2^-24 ulp of a / b: it can round the wrong way
    only where a / b is that close to a midpoint, that is where a 2^(k+1) - (2 n + 1) b = c for the quotient's
    integer n (24 bits; k = 23 or 24) and some |c| <= 4.  Those pairs are solved for and checked, for every
    29th odd b and those next to a power of two (all of them take 10 s and hold as well); an even b has the
    pairs of its odd part."""
    odd = np.arange((1 << 23) + 1, 1 << 24, 2, dtype=np.int64)
    B = np.concatenate([odd[::29], odd[:4096], odd[-4096:]])
    inv = B.copy()
    for _ in range(5):
        inv = (inv * (2 - B * inv)) & ((1 << 25) - 1)
    checked = 0
    for k in (23, 24):
        for c in (-3, -1, 1, 3):
            m = ((-c) * inv) & ((1 << (k + 1)) - 1)   # 2 n + 1, in [2^24, 2^25)
            if k == 23:
                m |= 1 << 24
            A = (m * B + c) >> (k + 1)
            ok = (m >= 1 << 24) & (m < 1 << 25) & (A >= 1 << 23) & (A < 1 << 24)
            a, b, n = A[ok], B[ok], m[ok] >> 1
            assert np.array_equal((a << (k + 1)) - (2 * n + 1) * b, np.full(a.shape, c))
            got, s = _markstein_quotient(a, b)
            want = (2 * (a << (47 - s)) + b) // (2 * b)
            inside = (want > (1 << 23) + 8) & (want < (1 << 24) - 8)      # (one spacing of results)
            assert np.array_equal(got[inside], want[inside]), (k, c)
            checked += int(inside.sum())
    assert checked > 400000
