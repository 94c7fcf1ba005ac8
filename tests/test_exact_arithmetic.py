"""The kernels' exact Case-1 arithmetic, modelled operation by operation on the host with the library's own
tables, against plain division and exact integers:
  - fl32(x / 10^a) by reciprocal and one residual: every 24-bit significand x and every a (falcon's FP32 and
    FP16 decode);
  - fl64(g / 10^a) for |g| < 2^32 by the 96-bit reciprocal, a <= 17 (FP64 decode);
  - the narrow test and g of an FP64 value with |v 10^a| < 10^8, a <= 13 (analysis, emit), and the FP32 ones."""
import os
import random
import re
import struct
from fractions import Fraction

import numpy as np
import pytest

M32, M64 = (1 << 32) - 1, (1 << 64) - 1
HEADER = os.path.join(os.path.dirname(__file__), "..", "paper_2511_04140_gb300", "csrc", "falcon_tables.h")


def table(name):
    body = re.search(r"%s\[\d+\] = \{(.*?)\};" % name, open(HEADER).read(), re.S).group(1)
    body = re.sub(r"/\*.*?\*/", "", body, flags=re.S)
    return [int(re.sub("[uUlL]+$", "", x.strip()), 0) for x in body.split(",") if x.strip()]


POW5, NORM, LOG2 = table("FALCON_POW5"), table("FALCON_POW5_NORM"), table("FALCON_LOG2_POW5")


def round_f32(a, b):
    """fl32(a + b) of FP64 values, rounded once: the sum is rounded to odd in FP64 first (two-sum)."""
    s = a + b
    t = s - a
    err = (a - (s - t)) + (b - t)
    s = np.where((err != 0) & ((err > 0) != (s > 0)), np.nextafter(s, 0.0), s)
    s = np.where(err != 0, (s.view(np.uint64) | np.uint64(1)).view(np.float64), s)
    return s.astype(np.float32)


@pytest.mark.parametrize("a", range(11))
def test_f32_quotient(a):
    p = np.float32(10.0 ** a)
    r = np.float32(1) / p
    for lo in range(1 << 23, 1 << 24, 1 << 21):
        x = np.arange(lo, lo + (1 << 21), dtype=np.float64)          # a power of two more or less changes nothing
        q = (x * float(r)).astype(np.float32).astype(np.float64)     # 48-bit products are exact in FP64
        e = (x - q * float(p)).astype(np.float32).astype(np.float64)
        got = round_f32(q, e * float(r))
        assert np.array_equal(got, x.astype(np.float32) / p)


@pytest.mark.parametrize("a", range(18))
def test_narrow_division(a):
    r2r1 = table("FALCON_RECIP5")[a] if a else M64
    r0, r1, r2 = np.uint64(table("FALCON_RECIP5_LO")[a]), np.uint64(r2r1 & M32), np.uint64(r2r1 >> 32)
    e0 = 11 - LOG2[a] - a + 52 + 1022 - 32
    rng = np.random.default_rng(a)
    near = [k * 5 ** a // 2 ** s + d for k in range(1, 200) for s in (0, 1, 2) for d in (-1, 0, 1)]
    g = np.concatenate([rng.integers(1, 1 << 32, 400_000), rng.integers(1, 1 << 20, 50_000), np.arange(1, 4096),
                        (1 << 32) - np.arange(1, 4096), 2 ** np.arange(32), [x for x in near if 0 < x < 1 << 32]]).astype(np.uint64)
    s = np.uint64(31) - np.floor(np.log2(g.astype(np.float64))).astype(np.uint64)
    u = np.uint64
    G = g << s
    lo = G * r1 + ((G * r0) >> u(32))
    T = G * r2 + (lo >> u(32))
    b = T >> u(63)
    M = ((T >> (u(9) + b)) + u(1)) >> u(1)
    top = (u(e0 - 1) - s + b << u(20)) + (M >> u(32))
    got = (top << u(32)) | (M & u(M32))
    assert np.array_equal(got.view(np.float64), g.astype(np.float64) / 10.0 ** a)


def passes(m, low, F, a):
    """Whether fl(round(m 5^a / 2^F) / 10^a) gives the value back: within half an ulp of it, scaled."""
    if F <= 0:
        return True
    d = (m * 5 ** a) % (1 << F)
    return 2 * ((1 << F) - d) <= 5 ** a if 2 * d >= 1 << F else (4 if m == low else 2) * d <= 5 ** a


def narrow_f64(u, a):
    """TestNarrow and Case1Narrow: (passes, |g|, left to the general test)."""
    hi, lo = u >> 32, u & M32
    e, mh = (hi >> 20) & 0x7FF, (hi & 0xFFFFF) | 0x100000
    top = (((mh << 32) | lo) << 11 >> 32) & M32
    sh = (1075 - a + 10 - LOG2[a] - 32 - 1 - e) & M32
    n = ((((top * (NORM[a] >> 32)) >> 32) >> sh if sh < 32 else 0) + 1) >> 1
    t = 6 if a < 3 else 0
    p5, lim = POW5[a] << t, (POW5[a] >> 1) << t
    f = (1075 - a + t - 32 - e) & M32
    P = (lo * p5 + (((mh * p5 - ((n << f) & M32 if f < 32 else 0)) & M32) << 32)) & M64
    return (P + lim) & M64 <= 2 * lim, n, f > 32


def narrow_f32(u, a):
    d = LOG2[a]
    P = (((u << 8) | 0x80000000) & M32) * (POW5[a] << (31 - d))
    lim = (POW5[a] >> 1) << (39 - d)
    sh = (150 - a + 7 - d - 1 - ((u >> 23) & 0xFF)) & M32
    n = (((P >> 32) >> sh if sh < 32 else 0) + 1) >> 1
    D = (P - (((n << (sh + 1)) & M32 if sh < 31 else 0) << 32) + lim) & M64
    return D <= 2 * lim and sh < 32, n


def candidates(rng, a, digits, limit):
    for _ in range(12_000):
        g = rng.randrange(1, 10 ** rng.randrange(1, digits + 1))
        yield from (Fraction(g, 10 ** a), Fraction(2 * g + 1, 2 * 10 ** a), rng.random() * Fraction(10) ** (rng.randrange(-6, digits) - a),
                    Fraction(2) ** rng.randrange(-40, limit.bit_length()))


@pytest.mark.parametrize("a", range(14))
def test_narrow_case1_f64(a):
    rng = random.Random(a)
    passed = 0
    for x in candidates(rng, a, 8, 10 ** 8):
        b = struct.unpack("<Q", struct.pack("<d", float(x)))[0] + rng.choice([0, 0, 1, -1, 2])
        v = Fraction(struct.unpack("<d", struct.pack("<Q", b))[0])
        if v * 10 ** a >= 10 ** 8:
            continue
        want = passes((b & ((1 << 52) - 1)) | 1 << 52, 1 << 52, 1075 - (b >> 52) - a, a)
        ok, n, left = narrow_f64(b, a)
        assert left or ok == want, (float(v), a)
        if want:
            assert n == int(v * 10 ** a + Fraction(1, 2)), (float(v), a)
        passed += want
    assert passed > 1000                           # both answers occur


@pytest.mark.parametrize("a", range(11))
def test_case1_f32(a):
    rng = random.Random(a)
    passed = 0
    for x in candidates(rng, a, 7, 10 ** 7):
        b = struct.unpack("<I", struct.pack("<f", float(x)))[0] + rng.choice([0, 0, 1, -1, 2])
        v = Fraction(struct.unpack("<f", struct.pack("<I", b))[0])
        if v * 10 ** a >= 10 ** 7 or b < 1 << 23:
            continue
        F = 150 - (b >> 23) - a
        want = F < 64 and passes((b & ((1 << 23) - 1)) | 1 << 23, 1 << 23, F, a)
        ok, n = narrow_f32(b, a)
        assert ok == want, (float(v), a)
        if want:
            assert n == int(v * 10 ** a + Fraction(1, 2)), (float(v), a)
        passed += want
    assert passed > 1000
