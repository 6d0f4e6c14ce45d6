"""The reciprocal root and exponential of the float64 pair forms (pair64.cuh)
next to powers of two, on the host.

PTX promises 2^-22.9 of rsqrt.approx, not where it lands: its result may be a
float32 step or more to the wrong side of a power of two, where the units of
the corrected value change.  pair64.cuh is compiled with g++ (its intrinsics
are IEEE operations) and every float32 within 2^-22.9 of the root is tried as
the approximation, for 32 float32 values on each side of every power of four in
the fast range and several low parts of r2.
Bounds: |h| < 2^-43 as the header states; 1/r to 1.5 units of 2^-53 relative to
the value (its rounding, and the square's r2 y in h); the Yukawa value e^(-k r)/r
to 2 (1 + k r) units of 2^-52 (an ulp of the exponential, the final product's
rounding and k times r's).

The exponential's tail, likewise: where subnormal() does not send a pair to the
TAIL form e^(-k r) has to be normal or round to zero, and the TAIL form has to
return the subnormal values, to half their spacing beside the bound above.
"""
import os
import subprocess

ROOT = os.path.dirname(os.path.dirname(os.path.abspath(__file__)))
CSRC = os.path.join(ROOT, "paper_2003_01833_gb300", "csrc")

CUDA = r"""
#pragma once
#include <initializer_list>
#include <math.h>
#include <stdint.h>
#include <stdio.h>
#include <string.h>
#define __device__
#define __forceinline__ inline
#define __restrict__
static struct { int x; } threadIdx;
template <class T, class U> T bits(U u) { T t; memcpy(&t, &u, sizeof t); return t; }
static inline uint32_t __float_as_uint(float x) { return bits<uint32_t>(x); }
static inline int __float_as_int(float x) { return bits<int>(x); }
static inline float __uint_as_float(uint32_t x) { return bits<float>(x); }
static inline double __longlong_as_double(long long x) { return bits<double>(x); }
static inline int __double2hiint(double x) { return (int)(bits<uint64_t>(x) >> 32); }
static inline int __double2loint(double x) { return (int)bits<uint64_t>(x); }
static inline double __hiloint2double(int h, int l) { return bits<double>((uint64_t)(uint32_t)h << 32 | (uint32_t)l); }
static inline float __fmul_rn(float a, float b) { return a * b; }
static inline float __fadd_rn(float a, float b) { return a + b; }
static inline float __fsub_rn(float a, float b) { return a - b; }
static inline float __fmaf_rn(float a, float b, float c) { return fmaf(a, b, c); }
static inline float __uint2float_rn(uint32_t x) { return (float)x; }
static inline float __int2float_rn(int x) { return (float)x; }
static inline int __float2int_rn(float x) { return (int)rintf(x); }
static inline uint32_t __funnelshift_l(uint32_t lo, uint32_t hi, int s) { return hi << s | lo >> (32 - s); }
static float seed;  // what rsqrt.approx returns
#define asm(...) y = seed
"""

MAIN = r"""
#include "pair64.cuh"
using namespace tagi::p64;
int main()
{
    const double k = 0.75;
    const Rate rate = make_rate(k);
    long n = 0;
    double eh = 0, er = 0, ey = 0;
    for (int p = -34; p <= 34; p++)
        for (int j = -32; j <= 32; j++) {
            const float rh = __uint_as_float(__float_as_uint((float)ldexp(1.0, 2 * p)) + j);
            for (uint64_t low : {0ull, 1ull, 0xfffffffull, 0x10000000ull, 0x1fffffffull}) {
                const double r2 = bits<double>(bits<uint64_t>((double)rh) + low);
                if (!fast_range(r2)) continue;
                const float near = (float)(1.0 / sqrt((double)rh));
                for (int step = -3; step <= 3; step++) {
                    seed = __uint_as_float(__float_as_uint(near) + step);
                    const long double approx = sqrtl((long double)rh) * seed;
                    if (fabsl(approx - 1.0L) > exp2l(-22.9L)) continue;
                    n++;
                    const Root R = root(r2);
                    const long double r = sqrtl((long double)r2);
                    eh = fmax(eh, fabs(R.h));
                    er = fmax(er, (double)fabsl(R.ri() * r - 1.0L) * 0x1p53);
                    if (k * (double)r > 700.0) continue;
                    const float h = small32(R.h);
                    const double v = exp_neg<false>(R.t, h, h, rate, kExp2Table.v) * R.y;
                    const long double exact = expl(-k * r) / r;
                    ey = fmax(ey, (double)(fabsl(v / exact - 1.0L) / (1.0L + k * r)) * 0x1p52);
                }
            }
        }
    // the tail: errors in units of the bounds
    double et = 0, eg = 0;
    for (double kt = 1e-9; kt < 1e10; kt *= 1.37) {
        const Rate rt = make_rate(kt);
        for (double x = 690.0; x < 790.0; x += 0.0137) {
            const double r2 = (x / kt) * (x / kt);
            if (!fast_range(r2)) continue;
            seed = (float)(1.0 / sqrt(r2));
            const Root R = root(r2);
            const float h = small32(R.h);
            const long double kr = kt * sqrtl((long double)r2), e = expl(-kr);
            const double tiny = subnormal(r2, rt) ? 0 : exp_neg<false>(R.t, h, 0.0f, rt, kExp2Table.v);
            if (!subnormal(r2, rt))
                et = fmax(et, (double)(fabsl(tiny - e) / (0x1p-1075L + (2.0L + 2.0L * kr) * 0x1p-52L * e)));
            if (subnormal(r2, rt) && (kr < 706.0L || kr > 790.0L)) et = INFINITY;
        }
        for (double x = 690.0; x < 790.0; x += 0.0137) {
            const double a = x / kt;
            const long double ka = (long double)kt * a, e = expl(-ka);
            const double g = exp_neg<true>(a, 0.0f, 0.0f, rt, kExp2Table.v);
            eg = fmax(eg, (double)(fabsl(g - e) / (0x1p-1075L + (2.0L + 2.0L * ka) * 0x1p-52L * e)));
        }
    }
    printf("%ld %.17g %.4g %.4g %.4g %.4g\n", n, eh, er, ey, et, eg);
    return 0;
}
"""


def test_root_and_exponential(tmp_path):
    (tmp_path / "cuda_runtime.h").write_text(CUDA)
    (tmp_path / "main.cpp").write_text(MAIN)
    exe = str(tmp_path / "pair64")
    subprocess.check_call(["g++", "-std=c++17", "-O1", "-w", "-ffp-contract=off", "-I", str(tmp_path), "-I", CSRC,
                           str(tmp_path / "main.cpp"), "-o", exe, "-lm"])
    n, h, ri, yukawa, tail, gauss = (float(v) for v in subprocess.check_output([exe], text=True, timeout=300).split())
    assert n > 40000
    assert h < 2.0 ** -43
    assert ri <= 1.5
    assert yukawa <= 2.0
    assert tail <= 1.0 and gauss <= 1.0
