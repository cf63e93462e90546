"""csrc/digits.h compiled for the host: the functions that the digit-product kernels run. The issuer's and
the drain warps' sequences of accumulator waits, restarts and hand-overs agree, cannot wait for one
another in a circle and keep every sum exact; digits represent an entry to 2^(e-64) at the scale that
scale_exp gives; exact sums are rounded to nearest even."""
from fractions import Fraction
import math
import random
import shutil
import struct
import subprocess

import numpy as np
import pytest

import test_exactsum as T

PROGRAM = r"""
#include <cstdio>
#include <cstring>
#include "digits.h"
using namespace fo;
int main(int argc, char** argv) {
    FILE* f = std::fopen(argv[2], "rb");
    FILE* g = std::fopen(argv[3], "wb");
    if (!std::strcmp(argv[1], "order")) {
        // the loops of k_dig_mma's issuer and drain warps
        for (int gs = 1; gs <= 2; ++gs)
            for (int cnt = 1; cnt <= 140; ++cnt) {
                std::fprintf(g, "%d %d", gs, cnt);
                for (int l = 0; l < cnt; ++l) {
                    const int ph = l & ((4 << gs) - 1);
                    for (int q = 0; q < 4; ++q) {
                        const int a = acc_order(q, acc_place(ph, gs), gs);
                        const bool beg = acc_begins(a, acc_place(ph, gs), gs), end = acc_ends(a, ph, 1 << 30, gs);
                        std::fprintf(g, " %d%d%d%d", a, beg && l > 0, beg || l == 0, end || l == cnt - 1);
                    }
                }
                std::fprintf(g, " |");
                for (int l = 0; l < cnt; ++l)
                    for (int x = 0; x < 4; ++x) {
                        const int a = acc_order(x, l, gs);
                        if (acc_ends(a, l, cnt, gs)) std::fprintf(g, " %d", a);
                    }
                std::fprintf(g, "\n");
            }
    } else if (!std::strcmp(argv[1], "digits")) {
        double x;
        int64_t e;
        while (std::fread(&x, 8, 1, f) == 1 && std::fread(&e, 8, 1, f) == 1) {
            const uint64_t u = digits_of(x, (int)e);
            std::fwrite(&u, 8, 1, g);
        }
    } else if (!std::strcmp(argv[1], "scale")) {
        double b;
        while (std::fread(&b, 8, 1, f) == 1) {
            const int64_t e = scale_exp(b);
            std::fwrite(&e, 8, 1, g);
        }
    } else {
        int64_t v[3];
        while (std::fread(v, 8, 3, f) == 3) {
            const double d = fixed_to_double(v[0], v[1], (int)v[2]);
            std::fwrite(&d, 8, 1, g);
        }
    }
    std::fclose(f);
    return std::fclose(g);
}
"""


@pytest.fixture(scope="module")
def run(tmp_path_factory):
    cxx = shutil.which("g++")
    if cxx is None:
        pytest.skip("no host compiler")
    d = tmp_path_factory.mktemp("digits")
    (d / "g.cpp").write_text(PROGRAM)
    subprocess.run([cxx, "-O2", "-std=c++17", "-I", T.CSRC, str(d / "g.cpp"), "-o", str(d / "g")], check=True)

    def call(what, data=b""):
        (d / "in").write_bytes(data)
        subprocess.run([str(d / "g"), what, str(d / "in"), str(d / "out")], check=True)
        return (d / "out").read_bytes()
    return call


def test_issue_and_drain_sequences(run):
    lines = run("order").decode().splitlines()
    assert len(lines) == 2 * 140
    for line in lines:
        issue, drain = line.split("|")
        gs, cnt, *ev = issue.split()
        gs, cnt, drain = int(gs), int(cnt), [int(a) for a in drain.split()]
        first = 4 if gs == 1 else 0   # orders of the low units are 4..7, of the high ones 0..3
        assert len(ev) == 4 * cnt
        done, drained, restarts, pairs = [0] * 4, [0] * 4, [0] * 4, [0] * 4
        at = 0   # drain warps' place in their list

        def drain_all():   # as far as the committed groups allow, in their order
            nonlocal at
            while at < len(drain) and drained[drain[at]] < done[drain[at]]:
                drained[drain[at]] += 1
                at += 1

        for l in range(cnt):
            block = [tuple(map(int, e)) for e in ev[4 * l:4 * l + 4]]
            assert sorted(b[0] for b in block) == [0, 1, 2, 3]
            for a, waits, fresh, ends in block:
                if waits:
                    restarts[a] += 1
                    drain_all()
                    # the wait ends: everything it needs was issued before it
                    assert drained[a] >= restarts[a]
                assert fresh == (waits or l == 0)
                pairs[a] = (0 if fresh else pairs[a]) + first + a + 1
                assert pairs[a] * 16 * 128 * 128 <= 2 ** 24   # exact in a float32 accumulator
                if ends:
                    done[a] += 1
        drain_all()
        assert at == len(drain) and drained == done
        assert [restarts[a] + 1 for a in range(4)] == done


def test_digits_and_scale(run):
    rng = random.Random(13)
    xs = [0.0, -0.0, 5e-324, -2.2e-308, 1e-300, 0.98, -0.98, 1.0, -1.0]
    xs += [rng.uniform(-1, 1) * 2.0 ** rng.randint(-80, 80) for _ in range(20000)]
    xs += [s * (1 - k * 2.0 ** -53) * 2.0 ** q for s in (1, -1) for k in range(40) for q in (-7, 0, 1, 9)]
    big = [abs(x) * f for x, f in zip(xs, [1.0, 1.0 + 2 ** -50, 3.7, 1e4] * len(xs))]
    big = [max(b, abs(x)) for b, x in zip(big, xs)]
    es = np.frombuffer(run("scale", np.array(big).tobytes()), dtype=np.int64)
    for b, e in zip(big, es):
        assert Fraction(b) < Fraction(99, 100) * Fraction(2) ** int(e)
        if b >= 1e-290:   # no more than a factor of about two too wide
            assert Fraction(b) >= Fraction(49, 100) * Fraction(2) ** int(e)
    data = b"".join(struct.pack("<dq", x, int(e)) for x, e in zip(xs, es))
    us = np.frombuffer(run("digits", data), dtype=np.uint64)
    for x, e, u in zip(xs, es, us):
        v = sum(((int(u) >> (8 * (7 - p)) & 255) - 128) * Fraction(2) ** (-7 - 8 * p) for p in range(8))
        assert abs(v * Fraction(2) ** int(e) - Fraction(x)) <= Fraction(2) ** (int(e) - 64)
    inf = np.frombuffer(run("scale", np.array([math.inf, math.nan, 1.79e308]).tobytes()), dtype=np.int64)
    assert list(inf) == [1 << 20] * 3


def test_fixed_point_rounding(run):
    rng = random.Random(14)
    vs = [(0, 0, 0), (1, -(2 ** 32), 0), (0, 1, 0), (0, -1, -3), (2 ** 62, 2 ** 62, 0), (-(2 ** 62), -(2 ** 62), 4)]
    for _ in range(20000):
        hi = rng.getrandbits(rng.randint(1, 60)) * rng.choice([1, -1])
        lo = rng.getrandbits(rng.randint(1, 60)) * rng.choice([1, -1])
        if rng.random() < 0.3:   # ties and near ties
            hi = (rng.getrandbits(53) << 5 | rng.choice([16, 15, 17])) >> rng.randint(0, 3)
            lo = rng.choice([0, 1, -1])
        vs.append((hi, lo, rng.choice([0, 5, -9, 700, -700])))
    out = np.frombuffer(run("fixed", b"".join(struct.pack("<3q", *v) for v in vs)))
    for (hi, lo, e), d in zip(vs, out):
        assert float(d) == float(Fraction(hi * 2 ** 32 + lo) * Fraction(2) ** (e - 70))
