"""The hand-made conversions and the quotient of the field kernels, restated in FP32 and integer
operations and held to the FP64 unit's results: double -> float and integer -> double rounded
to nearest even (double_float_int, u64_double_int), and the FP64 quotient rounded to FP32
from pairs of floats (cg_quotient), whose result away from the middles between two floats must
be the rounded quotient and whose test for the middles must send every near one to the division."""
import numpy as np
import pytest

F = np.float32


def double_float_int(x):
    b = x.view(np.uint64)
    h, l = (b >> np.uint64(32)).astype(np.uint32), b.astype(np.uint32)
    e = ((h >> 20) & 0x7FF).astype(np.int64) - 896
    f = ((h & 0xFFFFF) << 3) | (l >> 29)
    r = l & 0x1FFFFFFF
    up = ((r > 0x10000000) | ((r == 0x10000000) & ((f & 1) == 1))).astype(np.uint32)
    got = ((h & 0x80000000) | (((e.astype(np.uint32) << np.uint32(23)) | f) + up)).view(F)
    return got, (e >= 1) & (e <= 254)  # elsewhere the conversion instruction


def u64_double_int(x):
    out = np.zeros(x.size)
    for k, v in enumerate(x.tolist()):
        if v:
            lz = 64 - v.bit_length()
            m = (v << lz) & (2 ** 64 - 1)
            f, r = m >> 11, m & 0x7FF
            f += 1 if r > 0x400 or (r == 0x400 and f & 1) else 0
            out[k] = np.array([((1023 + 63 - lz - 1) << 52) + f], np.uint64).view(np.float64)[0]
    return out


def cg_quotient(a, b):
    """(result, taken): taken where the kernel does not divide."""
    A, B = a.view(np.uint64), b.view(np.uint64)
    ah, al = (A >> np.uint64(32)).astype(np.uint32), A.astype(np.uint32)
    bh, bl = (B >> np.uint64(32)).astype(np.uint32), B.astype(np.uint32)
    e = (ah >> 20).astype(np.int64) - (bh >> 20).astype(np.int64)
    xh = (np.uint32(0x3F800000) | ((ah & 0xFFFFF) << 3) | (al >> 29)).view(F)
    yh = (np.uint32(0x3F800000) | ((bh & 0xFFFFF) << 3) | (bl >> 29)).view(F)
    xl = (al & 0x1FFFFFFF).astype(F) * F(2.0 ** -52)
    yl = (bl & 0x1FFFFFFF).astype(F) * F(2.0 ** -52)
    d = np.float64
    inv = (1.0 / yh.astype(d)).astype(F)
    q0 = xh * inv
    r = (xh.astype(d) - q0.astype(d) * yh.astype(d)).astype(F)        # exact
    q1 = ((r + xl).astype(d) - q0.astype(d) * yl.astype(d)).astype(F) * inv
    q = q0 + q1
    rest = q1 - (q - q0)
    ulp = np.where(q >= 1, F(2.0 ** -23), F(2.0 ** -24)).astype(F)
    m = np.abs(rest)
    taken = (np.abs(m - F(0.5) * ulp) > F(2.0 ** -38)) & (np.abs(m - F(0.25) * ulp) > F(2.0 ** -38)) & (q > 0.5)
    return q * np.ldexp(F(1), e.astype(np.int32)), taken & (np.abs(e) < 120)


def _doubles(rng, n, lo=-60, hi=60):
    return np.ldexp(1.0 + rng.random(n), rng.integers(lo, hi, n))


def test_double_to_float():
    rng = np.random.default_rng(1)
    x = _doubles(rng, 200000, -120, 120) * rng.choice([-1.0, 1.0], 200000)
    f = x.astype(F).astype(np.float64)
    half = 0.5 * (f + np.nextafter(f.astype(F), F(np.inf)).astype(np.float64))  # exact middles
    near = half * (1 + rng.integers(-3, 4, half.size) * 2.0 ** -53)
    top = np.array([2.0 ** 127, 3.4028234e38, 1.1754944e-38, np.nextafter(2.0, 0.0), 2.0 - 2.0 ** -25])
    for v in (x, half, near, top):
        got, taken = double_float_int(np.ascontiguousarray(v))
        assert np.array_equal(got[taken], v[taken].astype(F))
        assert taken.mean() > 0.5


def test_integer_to_double():
    rng = np.random.default_rng(2)
    x = rng.integers(0, 2 ** 63, 20000, dtype=np.uint64) * np.uint64(2) + rng.integers(0, 2, 20000, dtype=np.uint64)
    x >>= rng.integers(0, 64, 20000, dtype=np.uint64)
    ties = (rng.integers(2 ** 52, 2 ** 53, 4000, dtype=np.uint64) << np.uint64(11)) + np.uint64(0x400)
    edge = np.array([0, 1, 2 ** 53 - 1, 2 ** 53 + 1, 2 ** 54 + 2, 2 ** 64 - 1, 2 ** 64 - 1024, 2 ** 64 - 1025], np.uint64)
    for v in (x, ties, ties + np.uint64(1), ties - np.uint64(1), edge):
        assert np.array_equal(u64_double_int(v), np.array([float(k) for k in v.tolist()]))


@pytest.mark.parametrize("near", [False, True])
def test_quotient(near):
    rng = np.random.default_rng(3)
    n = 400000
    b = _doubles(rng, n)
    if near:  # quotients within a few 2^-40 of the middle between two floats
        q = _doubles(rng, n, -3, 3).astype(F)
        mid = 0.5 * (q.astype(np.float64) + np.nextafter(q, F(np.inf)).astype(np.float64))
        a = b * (mid * (1.0 + rng.normal(0.0, 2.0 ** -41, n)))
    else:
        a = _doubles(rng, n)
    got, taken = cg_quotient(a, b)
    want = (a / b).astype(F)
    assert np.array_equal(got[taken], want[taken])
    assert near or taken.mean() > 0.99
