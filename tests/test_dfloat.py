"""The hi/lo arithmetic of the FP32 path on the host: dfloat.cuh compiled with
its CUDA intrinsics written out, against 113-bit sums.  The bounds are the
errors of the textbook forms (every operation renormalised, a running sum by
df_add, 1 / sqrt by one Newton step), which are computed beside them."""
import os
import shutil
import subprocess

import pytest

HERE = os.path.dirname(os.path.abspath(__file__))
HEADER = os.path.join(HERE, "..", "paper_1907_02289_gb300", "csrc", "dfloat.cuh")

PROGRAM = r"""
#include <algorithm>
#include <cmath>
#include <cstdio>
#include <random>
#include <vector>
#define __device__
#define __forceinline__ inline
static inline float __fadd_rn(float a, float b) { return a + b; }
static inline float __fsub_rn(float a, float b) { return a - b; }
static inline float __fmul_rn(float a, float b) { return a * b; }
static inline float __fmaf_rn(float a, float b, float c) { return fmaf(a, b, c); }
static float jitter = 0.f;  // the hardware estimate: within two units of the last place
static inline float rsqrtf(float x) { return (1.f / sqrtf(x)) * (1.f + jitter); }
#include "dfloat_host.h"
using namespace bh;
#if __SIZEOF_LONG_DOUBLE__ == 16 && __LDBL_MANT_DIG__ == 113
typedef long double Q;
#else
typedef __float128 Q;
#endif
static Q mag(Q x) { return x < 0 ? -x : x; }
static Q root(Q x) { Q y = std::sqrt((double)x); for (int k = 0; k < 3; ++k) y = (y + x / y) / 2; return y; }
static df split(double v) { const float h = (float)v; return {h, (float)(v - (double)h)}; }
static Q val(df a) { return (Q)a.hi + a.lo; }
static void report(const char* name, std::vector<double> a, std::vector<double> b) {
    std::sort(a.begin(), a.end());
    std::sort(b.begin(), b.end());
    for (double q : {0.5, 0.9, 0.99}) printf("%s %g %.6g %.6g\n", name, q, a[(size_t)(q * a.size())], b[(size_t)(q * b.size())]);
}
int main() {
    std::mt19937_64 g(1);
    std::uniform_real_distribution<double> U(0, 1);
    std::normal_distribution<double> G;
    for (int n : {60, 600, 3000}) {  // terms of either sign that cancel to about 1e-3
        std::vector<double> plain, sum;
        for (int t = 0; t < 4000; ++t) {
            std::vector<df> v;
            for (int k = 0; k < n / 2; ++k) {
                const double m = std::exp(3 * U(g));
                v.push_back(split(m));
                v.push_back(split(-m * (1 + 1e-3 * G(g))));
            }
            std::shuffle(v.begin(), v.end(), g);
            Q ref = 0;
            df a = {0.f, 0.f};
            df_sum s = {0.f, 0.f, 0.f};
            for (const df& x : v) {
                ref += val(x);
                a = df_add(a, x);
                df_accumulate(s, x);
            }
            plain.push_back((double)mag((val(a) - ref) / ref));
            sum.push_back((double)mag((val(df_total(s)) - ref) / ref));
        }
        report(("sum" + std::to_string(n)).c_str(), plain, sum);
    }
    std::vector<double> plain, sum;  // a node's mass: Mk + ((hi - Mk) + (lo + err)), as the moments keep it
    for (int t = 0; t < 20000; ++t) {
        Q ref = 0;
        float M = 0.f;
        df a = {0.f, 0.f};
        df_sum s = {0.f, 0.f, 0.f};
        for (int k = 0; k < 8; ++k) {
            const df x = split(1e-12 * (1 + U(g)));
            ref += val(x);
            M += x.hi;
            a = df_add(a, x);
            df_accumulate(s, x);
        }
        plain.push_back((double)mag(((Q)M + ((a.hi - M) + a.lo)) / ref - 1));
        sum.push_back((double)mag(((Q)M + ((s.hi - M) + (s.lo + s.err))) / ref - 1));
    }
    report("mass", plain, sum);
    plain.clear();
    sum.clear();
    for (int t = 0; t < 40000; ++t) {  // m / r^3
        jitter = (float)((2 * U(g) - 1) * 1.2e-7);
        df d[3];
        Q r2 = 0;
        for (df& x : d) {
            x = split(std::exp(8 * U(g)) * G(g));
            r2 += val(x) * val(x);
        }
        const df m = split(1e-12 * (1 + U(g)));
        const Q f = val(m) / (r2 * root(r2));
        const df o = df_add(df_add(df_mul(d[0], d[0]), df_mul(d[1], d[1])), df_mul(d[2], d[2]));
        const float y0 = rsqrtf(o.hi);
        const df p = df_mul(o, two_prod(y0, y0));
        const df y = fast_two_sum(y0, 0.5f * y0 * df_add({1.f, 0.f}, {-p.hi, -p.lo}).hi);
        plain.push_back((double)mag(val(df_mul(df_mul(m, y), df_mul(y, y))) / f - 1));
        const df z = df_rsqrt(df_norm2(d[0], d[1], d[2]));
        sum.push_back((double)mag(val(df_mul(df_mul(m, z), df_sqr(z))) / f - 1));
    }
    report("cube", plain, sum);
}
"""


def test_errors_are_no_larger_than_the_textbook_forms(tmp_path):
    if not shutil.which("g++"):
        pytest.skip("no g++")
    src = open(HEADER).read().replace("#include <cuda_runtime.h>", "")
    (tmp_path / "dfloat_host.h").write_text(src)
    (tmp_path / "t.cpp").write_text(PROGRAM)
    exe = str(tmp_path / "t")
    subprocess.run(["g++", "-O2", "-std=c++17", "-ffp-contract=off", str(tmp_path / "t.cpp"), "-o", exe], check=True)
    lines = subprocess.run([exe], check=True, capture_output=True, text=True).stdout.split("\n")
    seen = 0
    for name, q, plain, here in (x.split() for x in lines if x):
        assert float(here) <= float(plain), (name, q, plain, here)
        seen += 1
    assert seen == 15
