"""Group sums of csrc/exactsum.h (one rescaling per group, terms shifted without branches) against the
term-by-term form and math.fsum: the rows of test_exactsum (narrow and wide exponents, zeros,
subnormals, values near the largest float64), in groups of eight padded with zeros; and lane-strided
sums of groups brought to one exponent and added, as the kernels' warps do."""
import math
import os
import shutil
import subprocess

import numpy as np
import pytest

import test_exactsum as T

PROGRAM = r"""
#include <cstdio>
#include <cstdint>
#include <cstring>
#include <vector>
#include "exactsum.h"
using namespace fo;
int main(int argc, char** argv) {
    FILE* f = std::fopen(argv[1], "rb");
    FILE* g = std::fopen(argv[2], "wb");
    int64_t rows;
    if (std::fread(&rows, 8, 1, f) != 1) return 1;
    for (int64_t r = 0; r < rows; ++r) {
        int64_t n;
        if (std::fread(&n, 8, 1, f) != 1) return 1;
        std::vector<uint64_t> x(n + 7, 0);
        if ((int64_t)std::fread(x.data(), 8, n, f) != n) return 1;
        XAcc a{0, 0, 0}, b{0, 0, 0}, c{0, 0, 0};
        for (int64_t j = 0; j < n; ++j) xacc_add_abs(a, x[j]);
        for (int64_t j = 0; j < n; j += 8) xacc_add_abs_group<8>(b, x.data() + j);
        // two halves merged
        for (int64_t j = 8; j < n; j += 16) xacc_add_abs_group<8>(c, x.data() + j);
        XAcc d{0, 0, 0};
        for (int64_t j = 0; j < n; j += 16) xacc_add_abs_group<8>(d, x.data() + j);
        xacc_merge(c, d);
        // 32 lane-strided accumulators brought to the largest exponent and added
        XAcc lane[32], t{0, 0, 0};
        for (int l = 0; l < 32; ++l) {
            lane[l] = XAcc{0, 0, 0};
            for (int64_t j = l; j < n; j += 256) {
                uint64_t v[8];
                for (int u = 0; u < 8; ++u) v[u] = j + 32 * u < n ? x[j + 32 * u] : 0;
                xacc_add_abs_group<8>(lane[l], v);
            }
            t.e = lane[l].e > t.e ? lane[l].e : t.e;
        }
        for (int l = 0; l < 32; ++l) {
            xacc_align(lane[l], t.e);
            xacc_add_aligned(t, lane[l].lo, lane[l].hi);
        }
        double out[4] = {xacc_to_double(a), xacc_to_double(b), xacc_to_double(c), xacc_to_double(t)};
        std::fwrite(out, 8, 4, g);
    }
    std::fclose(f);
    std::fclose(g);
    return 0;
}
"""


def test_group_sums_round_like_fsum(tmp_path):
    cxx = shutil.which("g++")
    if cxx is None:
        pytest.skip("no host compiler")
    src, exe = tmp_path / "g.cpp", tmp_path / "g"
    src.write_text(PROGRAM)
    subprocess.run([cxx, "-O2", "-std=c++17", "-I", T.CSRC, str(src), "-o", str(exe)], check=True)
    data = T.rows(77) + [np.zeros(5), np.array([5e-324]), np.array([0.0, 1e308, 5e-324]), np.ones(9)]
    fin, fout = tmp_path / "in", tmp_path / "out"
    with open(fin, "wb") as f:
        f.write(np.int64(len(data)).tobytes())
        for x in data:
            f.write(np.int64(len(x)).tobytes() + np.ascontiguousarray(x, dtype=np.float64).tobytes())
    subprocess.run([str(exe), str(fin), str(fout)], check=True)
    out = np.fromfile(fout).reshape(-1, 4)
    for x, o in zip(data, out):
        try:
            ref = math.fsum(np.abs(x))
        except OverflowError:
            ref = math.inf
        assert np.all(o == ref)
