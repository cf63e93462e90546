"""Index arithmetic of the float64 digit products (csrc/gemm_digits.cu), restated: the staggered
restarts of the four accumulators keep every sum exact and every accumulator drained before it
restarts, the digits represent an entry to 2^(e-64), and the fixed-point sum is rounded correctly."""
import random
import struct
from fractions import Fraction

import pytest


def begins(a, l, gs):
    return l == 0 or ((l + (a << gs)) & ((4 << gs) - 1)) == 0


def ends(a, l, cnt, gs):
    return l == cnt - 1 or ((l + 1 + (a << gs)) & ((4 << gs) - 1)) == 0


def order(q, l, gs):
    qm = (1 << gs) - 1
    if ((l + 1) & qm) == 0:
        return ((4 - (((l + 1) >> gs) & 3)) + q) & 3
    if (l & qm) == 0 and l > 0:
        return ((4 - ((l >> gs) & 3)) + 1 + q) & 3
    return q


@pytest.mark.parametrize("gs,first", [(1, 4), (2, 0)])
def test_accumulator_restarts(gs, first):
    for cnt in range(1, 140):
        pairs, live, finished, restarts = [0] * 4, [False] * 4, [0] * 4, [0] * 4
        for l in range(cnt):
            seq = [order(q, l, gs) for q in range(4)]
            assert sorted(seq) == [0, 1, 2, 3]
            starting = [a for a in seq if begins(a, l, gs)]
            ending = [a for a in seq if ends(a, l, cnt, gs)]
            if l > 0:   # the restarted accumulator's MMAs come last, a finishing one's first
                assert len(starting) <= 1 and all(seq[3] == a for a in starting)
            if l < cnt - 1:
                assert len(ending) <= 1 and all(seq[0] == a for a in ending)
            for a in seq:
                if begins(a, l, gs):
                    assert not live[a]
                    if l > 0:
                        restarts[a] += 1
                        assert finished[a] >= restarts[a]   # drained once per restart
                    pairs[a], live[a] = 0, True
                pairs[a] += first + a + 1
                assert pairs[a] * 16 * 128 * 128 <= 2 ** 24   # exact in a float32 accumulator
                if ends(a, l, cnt, gs):
                    finished[a] += 1
                    live[a] = False
        assert not any(live)


def double_bits(x):
    return struct.unpack("<Q", struct.pack("<d", x))[0]


def digits(x, e):
    b = double_bits(x)
    ex = (b >> 52) & 0x7FF
    m = (b & ((1 << 52) - 1)) | ((1 << 52) if ex else 0)
    sh = (ex or 1) - 1012 - e
    v = m << min(sh, 10) if sh >= 0 else ((m + (1 << (-sh - 1))) >> -sh if sh > -55 else 0)
    if b >> 63:
        v = -v
    u = v + 0x8080808080808080
    assert 0 <= u < 1 << 64
    return [((u >> (8 * (7 - p))) & 255) - 128 for p in range(8)]


def test_digits():
    rng = random.Random(3)
    for t in range(20000):
        e = rng.choice([0, 1, -3, 7, 60])
        x = rng.uniform(-0.99, 0.99) * 2.0 ** (e + rng.choice([0, 0, -rng.randint(0, 70)]))
        if t % 50 == 0:
            x = rng.choice([0.99, -0.99, 0.0, 1e-300]) * (2.0 ** e if t % 100 else 1.0)
        if abs(x) >= 0.99 * 2.0 ** e and x not in (0.99 * 2.0 ** e, -0.99 * 2.0 ** e):
            continue
        got = sum(Fraction(d) / 2 ** (7 + 8 * i) for i, d in enumerate(digits(x, e))) * Fraction(2) ** e
        assert abs(got - Fraction(x)) <= Fraction(2) ** (e - 64)


def fixed_to_double(hi, lo, e):
    mask = (1 << 64) - 1
    l = (((hi << 32) & mask) + (lo & mask)) & mask
    h = ((hi >> 32) + (lo >> 63) + (1 if l < (lo & mask) else 0)) & mask
    sign = h >> 63
    if sign:
        l = -l & mask
        h = (~h + (1 if l == 0 else 0)) & mask
    if not h | l:
        return 0.0
    lz = 64 - h.bit_length() if h else 128 - l.bit_length()
    if lz == 0:
        m, rest = h, l
    elif lz < 64:
        m, rest = ((h << lz) | (l >> (64 - lz))) & mask, (l << lz) & mask
    else:
        m, rest = (l << (lz - 64)) & mask, 0
    r, low = m >> 11, m & 0x7FF
    r += 1 if low > 0x400 or (low == 0x400 and (rest or r & 1)) else 0
    exp = 127 - lz + e - 70 + 1023
    assert 0 < exp < 2046
    return struct.unpack("<d", struct.pack("<Q", (((exp << 52) + r - (1 << 52)) & mask) | (sign << 63)))[0]


def test_fixed_point_rounding():
    rng = random.Random(4)
    for _ in range(20000):
        hi = rng.getrandbits(rng.randint(1, 60)) * rng.choice([1, -1])
        lo = rng.getrandbits(rng.randint(1, 60)) * rng.choice([1, -1])
        if rng.random() < 0.2:   # ties and near ties
            hi = (rng.getrandbits(53) << 5 | rng.choice([16, 15, 17])) >> rng.randint(0, 3)
            lo = rng.choice([0, 1, -1])
        e = rng.choice([0, 5, -9])
        assert fixed_to_double(hi, lo, e) == float(Fraction(hi * 2 ** 32 + lo) * Fraction(2) ** (e - 70))
