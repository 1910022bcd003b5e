"""The two-word whole-number sums of the dynamically ordered H.v launches
(csrc/two_word.cuh), compiled for the host: exact totals in any order, for as many equal
tiles as the largest sector has (2^32 rows in tiles of 32), and for terms of both signs."""
import os
import shutil
import subprocess

import pytest

ROOT = os.path.dirname(os.path.dirname(os.path.abspath(__file__)))
CSRC = os.path.join(ROOT, "paper_2605_26261_gb300", "csrc")

SOURCE = r"""
#include <cstdint>
#include <cstdio>
#include <cstdlib>
#include <initializer_list>
#include "two_word.cuh"
using namespace ftlm;
using i128 = __int128;

// 2^-40 units of a, as the kernels take a term
static i128 units40(double a, double scale)
{
    long long w[2] = {0, 0};
    if (!two_word_add(w, a, scale)) std::exit(3);
    return ((i128)w[0] << 40) + w[1];
}
static double value(i128 v, double unscale)  // v 2^-40 units, rounded once
{
    const long long hi = (long long)(v >> 40), lo = (long long)(v - ((i128)hi << 40));
    return ((double)hi + (double)lo * 0x1p-40) * unscale;
}

int main()
{
    const int warps = 1216;
    static long long w[warps][2];
    auto total = [&](double want, const char *what) {
        long long hi = 0, lo = 0;
        for (auto &p : w) {
            hi += p[0];
            lo += p[1];
            p[0] = p[1] = 0;
        }
        const double got = two_word_value(hi, lo, 1.0);
        if (got != want) {
            std::printf("%s: %.17g, not %.17g\n", what, got, want);
            std::exit(1);
        }
    };
    // equal terms of either sign whose rest is close to half a unit, dealt to the warps
    // evenly, all to one warp, and unevenly
    for (double a : {7492.4921875, -7492.4921875, 0.46875}) {
        const uint32_t n = a == 0.46875 ? 1u << 27 : 1u << 25;
        const double want = value(n * units40(a, 1.0), 1.0);
        for (uint32_t t = 0; t < n; ++t) two_word_add(w[t % warps], a, 1.0);
        total(want, "even");
        for (uint32_t t = 0; t < n; ++t) two_word_add(w[5], a, 1.0);
        total(want, "one warp");
        for (uint32_t t = 0; t < n; ++t) two_word_add(w[t % 7 ? 3 : t % warps], a, 1.0);
        total(want, "uneven");
    }
    // terms of both signs and all sizes, in two orders
    static double a[1 << 20];
    uint64_t s = 1;
    i128 sum = 0;
    for (double &v : a) {
        s = s * 6364136223846793005ull + 1442695040888963407ull;
        v = (double)(int64_t)s * 0x1p-63 * (double)(1ull << (s >> 59));
        sum += units40(v, 1024.0);
    }
    const int n = 1 << 20;
    for (int t = 0; t < n; ++t) two_word_add(w[t % 11], a[t], 1024.0);
    total(value(sum, 1.0), "order 1");
    for (int t = 0; t < n; ++t) two_word_add(w[(t * 7) % warps], a[n - 1 - t], 1024.0);
    total(value(sum, 1.0), "order 2");
    for (double bad : {(double)NAN, 1e300, -1e300, (double)INFINITY, -(double)INFINITY}) {
        long long p[2] = {0, 0};
        if (two_word_add(p, bad, 1.0)) std::exit(2);
    }
    std::puts("ok");
}
"""


@pytest.mark.skipif(shutil.which("g++") is None, reason="needs g++")
def test_two_word_sums_are_exact(tmp_path):
    src, exe = tmp_path / "two_word.cpp", tmp_path / "two_word"
    src.write_text(SOURCE)
    subprocess.run(["g++", "-O2", "-std=c++17", "-ffp-contract=off", "-x", "c++", "-I", CSRC, str(src), "-o", str(exe)],
                   check=True)
    r = subprocess.run([str(exe)], capture_output=True, text=True)
    assert r.returncode == 0 and r.stdout.strip() == "ok", (r.returncode, r.stdout)
