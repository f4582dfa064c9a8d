"""The short FP64 root and quotient of the QR chains (csrc/fast_fp64.cuh), compiled for the host with the device
functions they use: within one unit in the last place of the correctly rounded value over the exponents they take
themselves, for every reciprocal square root that its documented error (2 units) allows, and equal to it where they
hand over to the library (extreme exponents, zero, subnormal, infinite, NaN, negative)."""
import os
import subprocess

import paper_1802_06177_gb300

SOURCE = r"""
#include <cmath>
#include <cstdint>
#include <cstdio>
#include <cstring>
#include <limits>
#include <random>
#define __device__
#define __forceinline__ inline
template <class A, class B> static B as(A a) { B b; std::memcpy(&b, &a, sizeof b); return b; }
static int __double2hiint(double x) { return (int)(as<double, int64_t>(x) >> 32); }
static int __double2loint(double x) { return (int)as<double, int64_t>(x); }
static double __hiloint2double(int h, int l) { return as<uint64_t, double>(((uint64_t)(uint32_t)h << 32) | (uint32_t)l); }
static float __int_as_float(int i) { return as<int, float>(i); }
static uint32_t __float_as_uint(float f) { return as<float, uint32_t>(f); }
static int off;  // units in the last place that the reciprocal root is off by
static float rsqrtf(float x) { return as<uint32_t, float>(as<float, uint32_t>((float)(1.0 / std::sqrt((double)x))) + off); }
static float __frcp_rn(float x) { return (float)(1.0 / (double)x); }
using std::fma;
using std::sqrt;
#include "fast_fp64.cuh"
static int64_t ulps(double a, double b) {
    if (std::isnan(a) || std::isnan(b)) return std::isnan(a) && std::isnan(b) ? 0 : 1 << 30;
    int64_t d = as<double, int64_t>(a) - as<double, int64_t>(b);
    return d < 0 ? -d : d;
}
int main() {
    std::mt19937_64 g(1);
    auto value = [&](int lo, int hi) {
        uint64_t m = g() >> 12;
        if (g() % 8 == 0) m = g() % 2 ? m & 7 : ~(m & 7) & 0xfffffffffffffull;  // near a power of two
        return as<uint64_t, double>((uint64_t)(1023 + lo + (int)(g() % (uint64_t)(hi - lo + 1))) << 52 | m);
    };
    int64_t root = 0, quot = 0, edge = 0;
    for (int i = 0; i < 3000000; ++i) {
        const bool wide = i % 3 == 0;
        off = (int)(g() % 5) - 2;
        const double a = wide ? value(-900, 900) : value(-8, 8);
        root = std::max(root, ulps(slmc::fast_sqrt(a), std::sqrt(a)));
        double n = wide ? value(-400, 400) : value(-4, 4), d = wide ? value(-400, 400) : value(-4, 4);
        if (g() & 1) n = -n;
        if (g() & 1) d = -d;
        quot = std::max(quot, ulps(slmc::fast_div(n, d), n / d));
        const double x = value(g() & 1 ? 895 : -905, g() & 1 ? 905 : 895), y = value(-405, 405);
        root = std::max(root, ulps(slmc::fast_sqrt(x), std::sqrt(x)));
        quot = std::max(quot, ulps(slmc::fast_div(y, d), y / d));
        quot = std::max(quot, ulps(slmc::fast_div(n, y), n / y));
    }
    const double inf = std::numeric_limits<double>::infinity(), nan = std::numeric_limits<double>::quiet_NaN();
    const double special[] = {0.0, -0.0, 1.0, -1.0, 5e-324, -2e-310, 2.3e-308, 1.7e308, -1.7e308, inf, -inf, nan, 0x1p401, 0x1p-401,
                              0x1p901, 0x1p-901};
    for (double a : special) {
        edge = std::max(edge, ulps(slmc::fast_sqrt(a), std::sqrt(a)));
        for (double b : special) edge = std::max(edge, ulps(slmc::fast_div(a, b), a / b));
    }
    std::printf("%lld %lld %lld\n", (long long)root, (long long)quot, (long long)edge);
}
"""


def test_root_and_quotient_within_one_unit(tmp_path):
    src = tmp_path / "fast.cpp"
    src.write_text(SOURCE)
    csrc = os.path.join(os.path.dirname(paper_1802_06177_gb300.__file__), "csrc")
    subprocess.run(["g++", "-O2", "-std=c++17", "-ffp-contract=off", "-I", csrc, str(src), "-o", str(tmp_path / "fast")],
                   check=True)
    out = subprocess.run([str(tmp_path / "fast")], check=True, capture_output=True, text=True).stdout
    root, quot, edge = (int(v) for v in out.split())
    assert root <= 1 and quot <= 1 and edge == 0, out
