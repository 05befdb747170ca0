"""The Leduc kernels' split of a pair's hands into segments (segments.h, plain C++):
the search by wave count finds the smallest estimate of all numbers of segments, in the
fewest waves that reach it and with the most segments of these."""
import os
import subprocess

ROOT = os.path.dirname(os.path.dirname(os.path.abspath(__file__)))

PROGRAM = r"""
#include <cstdio>
#include <random>
#include "segments.h"
static int64_t every(int32_t pairs, int64_t n, int sm, int64_t lo, int64_t hi, double phase, double tile, double rows) {
    const double share[8] = {1.0, 1.0, 0.8, 0.6, 0.4, 0.25, 0.1, 0.05};
    double best = 1e300;
    int64_t at = lo;
    for (int64_t seg = lo; seg <= hi; ++seg) {
        const int64_t per = (n + seg - 1) / seg;
        double c = 0.0;
        for (double s : share) c += phase + tile * (double)(int64_t)((double)per * s / rows + 0.999);
        c *= (double)(((int64_t)pairs * seg + sm - 1) / sm);
        const auto waves = [&](int64_t q) { return ((int64_t)pairs * q + sm - 1) / sm; };
        if (c < best || (c == best && waves(seg) == waves(at))) { best = c; at = seg; }
    }
    return at;
}
int main() {
    std::mt19937_64 r(1);
    auto log_of = [&](double lo, double hi) { return std::exp(std::uniform_real_distribution<>(std::log(lo), std::log(hi))(r)); };
    for (int i = 0; i < 20000; ++i) {
        const int32_t pairs = (int32_t)log_of(1, 20000);
        const int64_t n = (int64_t)log_of(1, 3e6), lo = (n + 8191) / 8192;
        const int sm = i % 3 ? 152 : 1 + (int)(r() % 160);
        const int64_t hi = lo + (int64_t)(r() % 500);
        const double rows = i % 2 ? 128.0 : 256.0;
        const int64_t a = malib::cheapest_segments(pairs, n, sm, lo, hi, 5.0, 2.2, rows);
        const int64_t b = every(pairs, n, sm, lo, hi, 5.0, 2.2, rows);
        if (a != b) { std::printf("%d pairs, %lld hands, %d SMs, %lld..%lld: %lld, not %lld\n", pairs, (long long)n, sm,
                                  (long long)lo, (long long)hi, (long long)a, (long long)b); return 1; }
    }
    return 0;
}
"""


def test_search_by_waves_is_exhaustive(tmp_path):
    src, exe = tmp_path / "t.cpp", tmp_path / "t"
    src.write_text("#include <cmath>\n" + PROGRAM)
    subprocess.run(["g++", "-O2", "-std=c++17", "-ffp-contract=off", "-I", os.path.join(ROOT, "paper_2106_07551_gb300", "csrc"),
                    str(src), "-o", str(exe)], check=True)
    r = subprocess.run([str(exe)], capture_output=True, text=True, timeout=120)
    assert r.returncode == 0, r.stdout
