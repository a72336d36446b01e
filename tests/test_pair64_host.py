"""The pair weights of csrc/pair64.cuh (host path: the same bits as the device but
for the FP32 starting value) against 113-bit arithmetic. Two roundings of half a
unit and dropped terms below 2^-56 of the result: 1.1 ulp."""
import os
import subprocess

ROOT = os.path.dirname(os.path.dirname(os.path.abspath(__file__)))
SOURCE = r"""
#include <cmath>
#include <cstdio>
#include <random>
#include "paper_1007_3458_gb300/csrc/pair64.cuh"
using namespace qym::p64;
#if defined(__x86_64__)
typedef __float128 Q;
extern "C" __float128 sqrtq(__float128);
static Q root(Q x) { return sqrtq(x); }
#else
typedef long double Q;  // binary128 on AArch64
static Q root(Q x) { return sqrtl(x); }
#endif
static double ulps(double a, Q ref) {
    Q d = (Q)a - ref;
    if (d < 0) d = -d;
    return (double)(d / ((Q)std::nextafter((double)ref, INFINITY) - (Q)(double)ref));
}
int main() {
    std::mt19937_64 r(3);
    std::uniform_real_distribution<double> U(-1, 1), V(0, 1);
    double w3 = 0, w1 = 0;
    long n = 0, bad = 0;
    for (long it = 0; it < 400000; ++it) {
        const double sj = std::exp2(U(r) * (it % 11 == 0 ? 19 : 4));
        double xi[3], xj[3];
        for (int c = 0; c < 3; ++c) {
            xi[c] = U(r);
            xj[c] = it % 3 == 0 ? U(r) * sj : xi[c] + U(r) * std::exp2(-V(r) * 24);
        }
        if (it % 6 == 3) xi[2] = xj[2] = 0;
        if (it % 6 == 4) xj[0] = xi[0];
        const double g = it % 7 == 0 ? std::exp2(-(double)(it % 40)) : std::exp2(-V(r) * 60);
        F3 d[3];
        Q q2 = 0;
        for (int c = 0; c < 3; ++c) {
            d[c] = diff(split3(xi[c]), split3(xj[c]));
            const Q dd = (Q)xi[c] - (Q)xj[c];
            q2 += dd * dd;
        }
        const F3 r2 = norm2(d[0], d[1], d[2]);
        if (!r2_fits(r2.h) || !g_fits((float)g)) continue;
        const float y0 = (float)(1.0 / std::sqrt((double)r2.h) * (1 + U(r) * std::exp2(-22.0)));
        double a;
        if (g_over_r3(split3(g), r2, y0, 0, a)) w3 = std::fmax(w3, ulps(a, (Q)g / (q2 * root(q2))));
        w1 = std::fmax(w1, ulps(inv_r(r2, y0, 0), 1 / root(q2)));
        ++n;
    }
    for (long i = 0; i < 400000; ++i) {  // the split is exact
        const double x = U(r) * std::exp2((double)((long)(r() % 214) - 87));
        if (std::fabs(x) < std::exp2(-88.) || std::fabs(x) >= std::exp2(127.)) continue;
        const F3 s = split3(x);
        bad += (Q)s.h + (Q)s.m + (Q)s.l != (Q)x;
    }
    std::printf("%ld %.4f %.4f %ld\n", n, w3, w1, bad);
}
"""


def test_weights_within_an_ulp(tmp_path):
    src, exe = tmp_path / "p.cpp", tmp_path / "p"
    src.write_text(SOURCE)
    quad = ["-lquadmath"] if os.uname().machine == "x86_64" else []
    subprocess.run(["g++", "-O2", "-std=gnu++17", "-ffp-contract=off", "-I", ROOT, str(src), "-o", str(exe), *quad],
                   check=True)
    n, w3, w1, bad = subprocess.run([str(exe)], capture_output=True, text=True, check=True).stdout.split()
    assert int(n) > 100000 and int(bad) == 0
    assert float(w3) <= 1.1 and float(w1) <= 1.1, (w3, w1)
