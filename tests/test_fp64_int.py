"""The FP64 roots and reciprocals on the integer pipe (csrc/fp64_int.cuh), run
on the host against long double: k / sqrt(x), which every HLLC sound speed
takes, 1 / sqrt(x) and 1 / b, over all binades, mantissas at the ends of a
binade, both parities of the exponent and factors k on both sides of the
product's carry.  The seeds are the exact value cut to 21 mantissa bits and off
by up to 2^-20.

Bounds as the header derives them: half an ulp for the rounding, 2^-56 and the
dropped partial products before it: 0.6 ulp for the reciprocal and the root;
0.65 ulp with the factor, whose product is rounded from a mantissa one bit
shorter when it carries."""

import os
import subprocess

from test_plan2d import CSRC, CUDA, needs_gxx

PROGRAM = r"""
#include <cmath>
#include <cstdio>
#include <cstring>
#include <random>
#include "fp64_int.cuh"
using namespace hydro;
static uint64_t bits(double x) { uint64_t b; std::memcpy(&b, &x, 8); return b; }
static double dbl(uint64_t b) { double x; std::memcpy(&x, &b, 8); return x; }
static double worst[3];
static void note(int which, double got, long double want)
{
    int e;
    std::frexp(got, &e);
    const double err = (double)(std::fabs((long double)got - want) / std::ldexp(1.0L, e - 53));
    if (!(err <= worst[which])) worst[which] = err;
}
int main()
{
    std::mt19937_64 rng(3);
    const double gammas[] = {1.0000001, 1.01, 1.4, 5.0 / 3.0, 2.0, 3.9, 3.9999999, 4.0, 4.1, 16.0, 1e6};
    for (int n = 0; n < 2000000; ++n) {
        uint64_t m = rng() & ((1ull << 52) - 1);
        if (n % 8 == 1) m &= 0xffff;
        if (n % 8 == 2) m |= ((1ull << 52) - 1) & ~0xffffull;
        if (n % 64 == 3) m = 0;
        if (n % 64 == 4) m = (1ull << 52) - 1;
        const uint64_t e = n % 2 ? 1 + rng() % 2046 : 1018 + rng() % 10;
        const double x = dbl((e << 52) | m);
        // the hardware seed: 21 bits of the mantissa, here with an error on either side
        const auto seed = [&](long double v) {
            const double s = (double)(v * (1.0L + std::ldexp((long double)((int64_t)(rng() % 2001) - 1000) / 1000.0L, -20)));
            return (uint32_t)(bits(s) >> 32);
        };
        const long double root = 1.0L / std::sqrt((long double)x);
        note(1, dbl(rsqrt_bits(bits(x), seed(root))), root);
        const double k = std::sqrt(n % 3 ? gammas[n % 11] : std::ldexp(1.0 + (double)(rng() % 4096) / 4096.0, (int)(rng() % 8) - 4));
        const long double scaled = (long double)k * root;
        note(2, dbl(rsqrt_scaled_bits(bits(x), seed(root), bits(k))), scaled);
        if (e >= 2 && e <= 2040) {
            const double b = n % 3 ? x : -x;
            note(0, dbl(rcp_bits(bits(b), seed(1.0L / (long double)b))), 1.0L / (long double)b);
        }
    }
    std::printf("%.4f %.4f %.4f\n", worst[0], worst[1], worst[2]);
}
"""


@needs_gxx
def test_integer_pipe_accuracy(tmp_path):
    src, exe = str(tmp_path / "t.cpp"), str(tmp_path / "t")
    with open(src, "w") as f:
        f.write(PROGRAM)
    subprocess.run(["g++", "-std=c++17", "-O1", "-I", CSRC, "-I", os.path.join(CUDA, "include"), src, "-o", exe], check=True)
    r = subprocess.run([exe], capture_output=True, text=True, check=True, timeout=300)
    rcp, root, scaled = (float(v) for v in r.stdout.split())
    assert rcp <= 0.6 and root <= 0.6 and scaled <= 0.65, r.stdout
