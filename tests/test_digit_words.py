"""The digit slicing of the tensor-core products as the kernels do it (no GPU): a value
v below 2^e becomes the integer X = round(v 2^(55 - e)), whose bytes with a bias of
128 each are its seven base-256 digits.  The double-float form of X is emulated
operation by operation in exactly rounded binary32 (its carries run modulo 2^32),
the binary64 one in integers.  Checked: digits in [-128, 127] and the first in
[-128, 128], so that each is exact in f16 (and 1024 + 128 + d is, on the way); the
reconstruction to 0.52 units of X; and that the accumulators of the issue table in
rgf_tc.cuh stay below 2^24 where they have to be exact."""
import re
import struct
from fractions import Fraction
from pathlib import Path

import numpy as np

SRC = (Path(__file__).resolve().parents[1] / "paper_1107_5300_gb300" / "csrc" / "rgf_tc.cuh").read_text()
M = Fraction(12582912)
MASK = 0xFFFFFFFF


def rn32(x):
    """Nearest binary32 of a rational (ties to even), as a rational."""
    if x == 0:
        return Fraction(0)
    a = abs(x)
    e = a.numerator.bit_length() - a.denominator.bit_length()
    if a < Fraction(2) ** e:
        e -= 1
    ulp = Fraction(2) ** (max(e, -126) - 23)
    q = a / ulp
    n = q.numerator // q.denominator
    r = q - n
    if r > Fraction(1, 2) or (r == Fraction(1, 2) and n & 1):
        n += 1
    return n * ulp * (1 if x > 0 else -1)


def bits(x):
    return struct.unpack("<I", struct.pack("<f", float(x)))[0]


def words_df(h, l, e):
    s8 = Fraction(2) ** (15 - e)
    two22, two18 = Fraction(1 << 22), Fraction(1 << 18)
    t0 = rn32(h * s8 + M)
    r0 = rn32(h * s8 - rn32(t0 - M))
    t1 = rn32(r0 * two22 + M)
    r1 = rn32(r0 * two22 - rn32(t1 - M))
    z = rn32(rn32(l * s8) * two22)
    tz = rn32(z + M)
    rz = rn32(z - rn32(tz - M))
    t2 = rn32(rn32(r1 * two18 + rn32(rz * two18)) + M)
    i1 = (bits(t1) + bits(tz) - 0x96800000) & MASK
    i1 -= (i1 >> 31) << 32
    x = i1 * (1 << 18) + ((bits(t2) + 0x80808080 - 0x4B400000) & MASK)
    x &= (1 << 64) - 1
    return ((x >> 32) + ((bits(t0) << 8) & MASK) + 0x00808080 - 0x40000000) & MASK, x & MASK


def words_64(v, e):
    b = struct.unpack("<Q", struct.pack("<d", v))[0]
    E = (b >> 52) & 0x7FF
    x = 0
    if E not in (0, 2047):
        m, sh = (b & 0xFFFFFFFFFFFFF) | 1 << 52, E - 1020 - e
        x = m << sh if sh >= 0 else (m + (1 << (-sh - 1))) >> -sh if sh > -60 else 0
        x = -x if b >> 63 else x
    x = (x + 0x0080808080808080) & ((1 << 64) - 1)
    return x >> 32, x & MASK


def digits(hi, lo):
    return [(hi >> 16) - 128] + [((w >> s) & 255) - 128 for w, s in ((hi, 8), (hi, 0), (lo, 24), (lo, 16), (lo, 8), (lo, 0))]


def check(ds, v, e, units):
    assert -128 <= ds[0] <= 128 and all(-128 <= d <= 127 for d in ds[1:]), ds
    rec = sum(Fraction(d) * Fraction(2) ** (e - 7 - 8 * i) for i, d in enumerate(ds))
    assert abs(rec - v) <= Fraction(units) * Fraction(2) ** (e - 55), (float(v), e, float((rec - v) * Fraction(2) ** (55 - e)))


def values(rng, n):
    top = 1.0 - 2.0 ** -24
    yield from (0.0, top, -top, 0.5, -0.5, 2.0 ** -30, -(2.0 ** -40), 127.5 / 256, -128.5 / 256, 2.0 ** -55, -1.5 * 2.0 ** -55,
                0.5 + 2.0 ** -25, -(0.25 + 2.0 ** -26), 1.0 / 3, 2.0 ** -23 * 0.75, top - 2.0 ** -50, 2.0 ** -8 - 2.0 ** -52)
    for _ in range(n):
        yield float(rng.choice([-1, 1]) * rng.random() * 2.0 ** -rng.integers(0, 58))


def test_double_float_words():
    rng = np.random.default_rng(0)
    for i, f in enumerate(values(rng, 1500)):
        e = int(rng.integers(-30, 31))
        v = f * 2.0 ** e
        h = np.float32(v)
        l = np.float32(v - float(h))
        if i % 3 == 0:                          # the low part of a sum: any, up to half an ulp, either sign
            l = np.float32(float(np.spacing(np.abs(h))) * rng.uniform(-0.5, 0.5))
        if abs(float(h)) >= 2.0 ** e:
            continue
        h, l = Fraction(float(h)), Fraction(float(l))
        check(digits(*words_df(h, l, e)), h + l, e, 0.52)


def test_binary64_words():
    rng = np.random.default_rng(1)
    for f in values(rng, 3000):
        e = int(rng.integers(-90, 91))
        v = f * 2.0 ** e
        check(digits(*words_64(v, e)), Fraction(v), e, 0.5)
    v = (1.0 - 2.0 ** -53) * 2.0 ** 5           # every digit at its end
    check(digits(*words_64(v, 5)), Fraction(v), 5, 0.5)
    check(digits(*words_64(-v, 5)), Fraction(-v), 5, 0.5)


def const(name):
    return int(re.search(rf"constexpr int {name} = (\d+);", SRC).group(1))


def test_accumulators_hold_their_sums():
    S, real = const("S"), 2 * const("KGRP")
    table = re.search(r"kMma\[NMMA\] = \{(.*?)\};", SRC, re.S).group(1)
    ops = [tuple(map(int, t)) for t in re.findall(r"\{(\d+), (\d+), (\d+), (\d+)\}", table)]
    assert len(ops) == const("NMMA")
    level = {0: 0, 1: 1, 2: 2, 3: 3, 4: 4, 5: 5, 6: 6, 7: 4}
    seen, terms = set(), dict.fromkeys(level, 0)
    for i, j0, nd, acc in ops:
        for q in range(nd):
            assert (i, j0 + q) not in seen and level[acc + q] == i + j0 + q
            seen.add((i, j0 + q))
            terms[acc + q] += 1
    assert seen == {(i, j) for i in range(S) for j in range(S - i)}
    for acc, n in terms.items():
        if level[acc] <= 4:
            assert n * real * 128 * 128 <= 2 ** 24, acc
    # the rank-b update: one accumulator a level, 16 complex inner entries
    assert 5 * 32 * 128 * 128 <= 2 ** 24
