"""The bit conversions of the FP64 fine grid (dw.cuh: widen, narrow) against the casts, bit for bit,
over the exponent range with its ends, infinities, NaN and random patterns.  By design apart: widen
keeps subnormals below 2^-126 only, narrow gives 0 below 2^-126 and rounds halves away from zero."""
import os
import subprocess

ROOT = os.path.dirname(os.path.dirname(os.path.abspath(__file__)))

SRC = r"""
#include <math.h>
#include <stdint.h>
#include <stdio.h>
#include <string.h>
#include "dw.cuh"
static uint64_t g = 88172645463325252ull;
static uint64_t rnd() { g ^= g << 13; g ^= g >> 7; g ^= g << 17; return g; }
static long bad = 0;
template <class T> static bool same(T a, T b) { return (a != a && b != b) || memcmp(&a, &b, sizeof(T)) == 0; }
static const float least = 1.17549435e-38f;             // 2^-126
static void n(uint64_t u) {
    double d;
    memcpy(&d, &u, 8);
    float want = (float)d;
    if (fabs(d) < (double)least) want = copysignf(0.0f, (float)d);
    else if ((u & 0x1fffffff) == 0x10000000 && !(u >> 29 & 1)) want = nextafterf(want, copysignf(INFINITY, want));
    bad += !same(firm::narrow(d), want);
}
static void w(uint32_t b) {
    float v;
    memcpy(&v, &b, 4);
    const double d = firm::widen(v);
    bad += fabsf(v) < least ? !(fabs(d) <= (double)least) : !same(d, (double)v);
}
int main() {
    for (int i = 0; i < 1000000; ++i) {                 // integers of either sign at any unit
        const float v = (float)(int)((rnd() & 1 ? 1 : -1) * (1 + (int64_t)(rnd() >> (33 + rnd() % 31))));
        const int e = (int)(rnd() % 400) - 200;
        bad += !same(firm::widen_scaled(v, e), ldexp((double)v, e));
    }
    for (uint64_t e = 0; e < 2048; ++e)                 // every exponent, around the ends and ties of the mantissa
        for (uint64_t m : {0ull, 1ull, 0xfffffffull, 0x10000000ull, 0x10000001ull, 0x1fffffffull, 0x2fffffffull,
                           0x30000000ull, 0x30000001ull, 0xfffffe0000000ull, 0xfffffefffffffull, 0xffffff0000000ull,
                           0xfffffffffffffull})
            for (uint64_t s = 0; s < 2; ++s) n(s << 63 | e << 52 | m);
    for (uint32_t e = 0; e < 256; ++e)
        for (uint32_t m : {0u, 1u, 0x3fffffu, 0x400000u, 0x7fffffu})
            for (uint32_t s = 0; s < 2; ++s) w(s << 31 | e << 23 | m);
    for (int i = 0; i < 4000000; ++i) {
        n(rnd());
        n((rnd() & 0x800fffffffffffffull) | (870 + rnd() % 290) << 52);
        w((uint32_t)rnd());
    }
    printf("%ld\n", bad);
    return 0;
}
"""


def test_conversions_against_the_casts(tmp_path):
    src, exe = tmp_path / "conv.cu", tmp_path / "conv"
    src.write_text(SRC)
    csrc = os.path.join(ROOT, "paper_1307_5824_gb300", "csrc")
    from paper_1307_5824_gb300.build import nvcc
    subprocess.run([nvcc(), "-std=c++17", "-O1", "-gencode", "arch=compute_103a,code=sm_103a", "-I", csrc, str(src),
                    "-o", str(exe)], check=True, capture_output=True, text=True)
    out = subprocess.run([str(exe)], check=True, capture_output=True, text=True)
    assert out.stdout.strip() == "0"
