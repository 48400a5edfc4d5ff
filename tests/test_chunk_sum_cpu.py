"""The FP64 sum of FP32 values 16 at a time (csrc/chunk_sum.h, the slice sum's arithmetic)
against FP64 additions one by one, on the host: bit for bit where those never round, large
values that cancel and far smaller ones that stay among them, within one chunk and across
chunks; elsewhere no further from the exact sum than one rounding per value allows."""
import os
import shutil
import subprocess

import pytest

CSRC = os.path.join(os.path.dirname(os.path.dirname(os.path.abspath(__file__))), "paper_2112_15083_gb300", "csrc")

CHECK = r"""
#include <math.h>
#include <stdio.h>
#include <string.h>
#include <random>
#include <vector>
#include "chunk_sum.h"
static int bad = 0;
static long long exact_sums = 0;
static void check(const char *what, const std::vector<float> &v) {
    tnk::ChunkSum s;
    for (size_t i = 0; i < v.size(); i += 16) {
        float x[16];
        memcpy(x, &v[i], sizeof(x));
        s.add16(x);
    }
    double seq = 0, mag = 0, err = 0;  // err: the exact sum minus seq, from two-sums
    bool rounds = false;
    for (float y : v) {
        const double t = seq + y, b = t - seq, e = (seq - (t - b)) + (y - b);
        rounds |= e != 0;
        err += e;
        seq = t;
        mag += fabs((double)y);
    }
    const double got = s.total();
    bool ok;
    if (!std::isfinite(seq)) ok = std::isnan(seq) ? std::isnan(got) : got == seq;
    else if (!rounds) { ok = memcmp(&got, &seq, 8) == 0; exact_sums++; }
    else ok = fabs((got - seq) - err) <= v.size() * ldexp(mag, -53);
    if (!ok && ++bad <= 10) printf("%s: %.17g, one by one %.17g (rounds: %d)\n", what, got, seq, rounds);
}
static std::vector<float> chunks(std::vector<std::vector<double>> c) {
    std::vector<float> v;
    for (auto &x : c) {
        x.resize(16, 0.0);
        for (double y : x) v.push_back((float)y);
    }
    return v;
}
int main() {
    const double t45 = ldexp(1, -45), t75 = ldexp(1, -75), t50 = ldexp(1, -50), b20 = ldexp(1, 20);
    check("cancel, two tails", chunks({{1, -1, t45, t75}}));
    check("cancel across chunks", chunks({{b20}, {-b20, t45}}));
    check("tail first", chunks({{t45}, {-t45, 1, -1, t75}}));
    check("tail cancels", chunks({{t50}, {-t50, 8}, {-8, t75}}));
    check("tails of two chunks", chunks({{1, t50}, {-1, t45}, {-t45, ldexp(1, -60)}}));
    check("low kept, narrow chunks", chunks({{1, -1, 3, t45}, {2, 5}, {-10, t50}}));
    check("far down", chunks({{1, -1, ldexp(1, -110), ldexp(3, -125)}}));
    std::mt19937_64 g(5);
    auto below = [&](int n) { return (int)(g() % n); };
    // random sums that never round one by one: a value is taken if its addition is exact
    for (int it = 0; it < 60000; it++) {
        const int n = 16 * (1 + below(6)), spread = 1 + below(70), top = below(40) - 30;
        std::vector<float> v;
        double acc = 0;
        while ((int)v.size() < n) {
            float y = 0.f;
            for (int tries = 0; tries < 8; tries++) {
                const int bits = 1 + below(24);
                float c = ldexpf((float)(1 + below(1 << bits)), top - below(spread) - bits);
                if (below(2)) c = -c;
                if (below(4) == 0) c = -(float)acc;             // cancel what the sum holds
                if (below(4) == 0 && !v.empty()) c = -v[below((int)v.size())];
                const double t = acc + c, b = t - acc, e = (acc - (t - b)) + (c - b);
                if (e == 0) { y = c; acc = t; break; }
            }
            v.push_back(y);
        }
        check("random, exact one by one", v);
    }
    // sums that do round: any spread, gaps of zeros, infinities and NaN, the ends of the range
    std::normal_distribution<float> nd;
    for (int it = 0; it < 60000; it++) {
        std::vector<float> v(16 * (1 + below(20)));
        const int kind = below(8), spread = 1 + below(80), base = below(100) - 60;
        for (float &y : v) {
            y = ldexpf(nd(g), base - below(spread));
            switch (kind) {
                case 0: if (below(3) == 0) y = below(2) ? 0.f : -0.f; break;
                case 1: if (below(2)) y = ldexpf(y, -54); break;
                case 2: if (below(400) == 0) y = below(2) ? INFINITY : NAN; break;
                case 3: y = ldexpf(y, -100); break;
                case 4: y = ldexpf(nd(g), 118); break;
                case 5: y = ldexpf(nd(g), base); break;
            }
        }
        check("random", v);
    }
    printf("%d differ, %lld exact\n", bad, exact_sums);
    return bad != 0 || exact_sums < 60000;
}
"""


def test_chunk_sum_is_the_sum_one_by_one_where_that_is_exact(tmp_path):
    cxx = shutil.which("g++") or shutil.which("c++")
    if cxx is None:
        pytest.skip("no C++ compiler")
    src, exe = tmp_path / "c.cpp", tmp_path / "c"
    src.write_text(CHECK)
    subprocess.run([cxx, "-O2", "-std=c++17", "-ffp-contract=off", "-I", CSRC, str(src), "-o", str(exe)], check=True)
    r = subprocess.run([str(exe)], capture_output=True, text=True, timeout=300)
    assert r.returncode == 0, r.stdout + r.stderr
