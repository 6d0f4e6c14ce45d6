// Float64 kernel values of the plain form: 1/r, r and 2^v from the squared
// distance, for hardware whose float64 unit is 73 times slower than its
// float32 one.
//
// The SM retires 1.68 float64 operations a clock (a conversion between float32
// and float64 costs as much), against 123 of float32: one float64
// instruction of a warp takes as long as 70 others.  sqrt, exp and a division
// from the math library come to 47 such slots a pair with the rest of a
// Yukawa term.  Here a pair costs 8 for its geometry and 4 a field; the rest
// is float32 and integer work that hides behind them:
//   1/r   the float32 approximation of rsqrt corrected in two-float arithmetic
//         (y, to 2^-44), and its defect h = (1 - r2 y^2) / 2 in float64: 1/r =
//         y (1 + h) and r = r2 y (1 + h).  The series ends at 2^-86; the rounding
//         of r2 y leaves 2^-54 in h.  Ten bits of h are enough in the
//         exponential, and the factors go into its float32 part;
//   2^v   Tang's table-driven exponential (ACM TOMS 15, 1989): v = (n + f)/512,
//         2^v = 2^(n >> 9) T[n & 511] 2^(f/512), T in float64, the factor's
//         difference from 1 (below 2^-10) in two-float arithmetic, added to
//         T's mantissa as an integer.
// Every bit pattern below is that of IEEE 754 binary32 and binary64.
#pragma once

#include <cuda_runtime.h>
#include <stdint.h>

namespace tagi {
namespace p64 {

constexpr int kTab = 512;

// T[j] = 2^(j/512) rounded to nearest: powers of 2^(1/512) in double-double
// arithmetic (Dekker's product), at compile time.
struct Exp2Table {
    double v[kTab];
    static constexpr double split(double a)
    {
        const double t = 134217729.0 * a;  // 2^27 + 1
        return t - (t - a);
    }
    constexpr Exp2Table() : v()
    {
        const double gh = 0x1.0058c86da1c0ap+0, gl = -0x1.5e00e62d6b30dp-56;  // 2^(1/512)
        double h = 1.0, l = 0.0;
        for (int j = 0; j < kTab; j++) {
            v[j] = h;
            const double p = h * gh;
            const double a1 = split(h), a2 = h - a1, b1 = split(gh), b2 = gh - b1;
            const double e = ((a1 * b1 - p) + a1 * b2 + a2 * b1) + a2 * b2 + (h * gl + l * gh);
            h = p + e;
            l = e - (h - p);
        }
    }
};
static __device__ const Exp2Table kExp2Table = Exp2Table();

__device__ __forceinline__ void load_table(double* tab, int threads)
{
    for (int j = threadIdx.x; j < kTab; j += threads) tab[j] = kExp2Table.v[j];
}

// float32 truncation of a positive float64 in float32's range, and what it leaves
__device__ __forceinline__ float trunc32(int hi, uint32_t lo)
{
    return __uint_as_float(((uint32_t)(hi - 0x38000000) << 3) | (lo >> 29));
}

// whether r2 takes the fast path (2^-70 <= r2 < 2^70); zero, tiny, huge and
// non-finite values do not
__device__ __forceinline__ bool fast_range(double r2)
{
    return (uint32_t)(__double2hiint(r2) - 0x3B900000) < 0x44500000u - 0x3B900000u;
}

// 1/sqrt(r2) = y (1 + h) and sqrt(r2) = t (1 + h), |h| < 2^-43
struct Root {
    double y, t, h;
    __device__ __forceinline__ double ri() const { return fma(y, h, y); }
    __device__ __forceinline__ double r() const { return fma(t, h, t); }
};

__device__ __forceinline__ Root root(double r2)
{
    const int hi = __double2hiint(r2);
    const uint32_t lo = (uint32_t)__double2loint(r2);
    const float rh = trunc32(hi, lo);
    // the low 29 bits of the mantissa, units of 2^(exponent - 52)
    const float rl =
        __uint2float_rn(lo & 0x1fffffffu) * __uint_as_float((uint32_t)((hi & 0x7ff00000) - 0x3B400000) << 3);
    float y;
    asm("rsqrt.approx.ftz.f32 %0, %1;" : "=f"(y) : "f"(rh));
    // e = 1 - r2 y^2 to 2^-45
    const float p = __fmul_rn(y, y), pe = __fmaf_rn(y, y, -p);
    float e = __fmaf_rn(-rh, p, 1.0f);
    e = __fmaf_rn(-rh, pe, e);
    e = __fmaf_rn(-rl, p, e);
    const float yl = __fmul_rn(y, __fmul_rn(e, __fmaf_rn(0.375f, e, 0.5f)));
    // y + yl as a float64: yl in units of the last place of y's mantissa.  Where
    // that passes a power of two (the approximation may lie on either side of
    // one), the units beyond it are half, or twice, as large
    const uint32_t yb = __float_as_uint(y);
    const int q = __float2int_rn(yl * __uint_as_float((306u << 23) - (yb & 0x7f800000u)));
    const int64_t base = (int64_t)((yb >> 3) + 0x38000000u) << 32 | (uint32_t)(yb << 29);
    int64_t y64 = base + q;
    if (((uint32_t)(y64 >> 32) ^ (uint32_t)(base >> 32)) >> 20) {
        constexpr int64_t mantissa = (1ll << 52) - 1;
        y64 += q < 0 ? y64 - (base & ~mantissa) : -((y64 & mantissa) >> 1);
    }
    const double y0 = __longlong_as_double(y64);
    const double yhalf = __longlong_as_double(y64 - (1ll << 52));
    const double t = r2 * y0;
    return Root{y0, t, fma(-t, yhalf, 0.5)};
}

// 1/r and r within an ulp
__device__ __forceinline__ void inv_sqrt(double r2, double& ri, double& r)
{
    const Root R = root(r2);
    ri = R.ri();
    r = R.r();
}

// a float64 below 2^-40 in size, to float32's precision (zero stays zero)
__device__ __forceinline__ float small32(double h)
{
    const uint32_t hi = (uint32_t)__double2hiint(h), mag = hi & 0x7fffffffu;
    const uint32_t v = (mag - 0x38000000u) << 3 | (uint32_t)__double2loint(h) >> 29 | (hi & 0x80000000u);
    return mag < 0x38100000u ? 0.0f : __uint_as_float(v);
}

// Exponent factor of e^(-k a) = 2^(c a / 512): c = -512 k log2(e) as a
// float64, what the rounding left (a float32), and c as a float32; sub: see
// subnormal()
struct Rate {
    double c;
    float cl, cf;
    uint32_t sub;
};
__device__ __forceinline__ Rate make_rate(double k)
{
    constexpr double lh = 0x1.71547652b82fep+0, ll = 0x1.777d0ffda0d24p-56;  // log2(e)
    const double k5 = -512.0 * k, c = k5 * lh;
    const double r = 707.5 / k;  // e^-707.5 = 2^-1020.7
    return Rate{c, (float)(fma(k5, lh, -c) + k5 * ll), (float)c, (uint32_t)__double2hiint(r * r)};
}

// whether e^(-k r) may be below the normal range and not round to zero: 707.5 <=
// k r < 746, outwards, by the high word of r2 (the square of 746 / 707.5 is
// 1.112: at most 0.202 of a binade's 2^20 high words above)
__device__ __forceinline__ bool subnormal(double r2, const Rate& k)
{
    return (uint32_t)(__double2hiint(r2) - (int)k.sub) < 0x34000u;
}

// e^(-k a (1 + da)) (1 + h) for a >= 0 in float32's range and |da|, |h| < 2^-42,
// to an ulp beside the rounding of a.  Below 2^-1021: with TAIL rounded to a
// multiple of 2^-1074, without it 0 (a branch here costs a kernel of two fields
// 6%; its callers keep such pairs away, subnormal())
template <bool TAIL>
__device__ __forceinline__ double exp_neg(double a, float da, float h, const Rate& k, const double* __restrict__ tab)
{
    const float af = trunc32(__double2hiint(a), (uint32_t)__double2loint(a));
    // n = the integer nearest c a (from the float32 product; never positive)
    const float v = fmaxf(__fmul_rn(af, k.cf), -1.0e6f);
    const float nm = __fadd_rn(v, 12582912.0f);  // 1.5 * 2^23
    const int n = __float_as_int(nm) - 0x4B400000;
    // f + 3 in [2, 4): its mantissa is f in units of 2^-51
    const float n3 = __fsub_rn(3.0f, __fsub_rn(nm, 12582912.0f));  // 3 - n, an integer >= 3
    const uint32_t nb = __float_as_uint(n3);
    const double g = fma(a, k.c, __hiloint2double((int)((nb >> 3) + 0x38000000u), (int)(nb << 29)));
    const uint32_t ghi = (uint32_t)__double2hiint(g), glo = (uint32_t)__double2loint(g);
    const int fi = (int)(__funnelshift_l(glo, ghi, 12) ^ 0x80000000u);  // f in units of 2^-31, rounded down
    const float fh = __int2float_rn(fi & ~0x7f) * 0x1p-31f;             // 24 bits
    const float fl = __fmaf_rn(
        v, da, __fmaf_rn(af, k.cl, __uint2float_rn(((uint32_t)fi & 0x7fu) << 20 | (glo & 0xfffffu)) * 0x1p-51f));
    // P - h = 2^(f/512) - 1 = f (c1 + f (c2 + f (c3 + f c4))), c_i = (ln 2 / 512)^i / i!
    constexpr float c1h = 0x1.62e430p-10f, c1l = -0x1.05c610p-38f, c2h = 0x1.ebfbe0p-21f, c2l = -0x1.f4e9c6p-51f,
                    c3 = 0x1.c6b08ep-32f, c4 = 0x1.3b2ab6p-43f;
    const float w = __fmul_rn(fh, __fmaf_rn(fh, c4, c3));
    const float qh = __fadd_rn(c2h, w), ql = __fadd_rn(__fadd_rn(__fsub_rn(c2h, qh), w), c2l);
    const float sh = __fmul_rn(fh, qh);
    const float sl = __fmaf_rn(fl, qh, __fmaf_rn(fh, ql, __fmaf_rn(fh, qh, -sh)));
    const float ih = __fadd_rn(c1h, sh), il = __fadd_rn(__fadd_rn(__fsub_rn(c1h, ih), sh), __fadd_rn(sl, c1l));
    const float ph = __fmul_rn(fh, ih);
    const float pl = __fadd_rn(h, __fmaf_rn(fl, ih, __fmaf_rn(fh, il, __fmaf_rn(fh, ih, -ph))));
    // G = T P, |G| < 2^-9, added to T as an integer in units of 2^-52
    const double T = tab[n & (kTab - 1)];
    const int thi = __double2hiint(T);
    const uint32_t tlo = (uint32_t)__double2loint(T);
    const float th = trunc32(thi, tlo), tl = __uint2float_rn(tlo & 0x1fffffffu) * 0x1p-52f;
    const float Gh = __fmul_rn(th, ph);
    const float Gl = __fmaf_rn(tl, ph, __fmaf_rn(th, pl, __fmaf_rn(th, ph, -Gh)));
    const float m1 = __fadd_rn(Gh, 0x1.8p-8f);                                           // units of 2^-31
    const float m2 = __fadd_rn(__fadd_rn(__fsub_rn(Gh, __fsub_rn(m1, 0x1.8p-8f)), Gl), 0x1.8p-29f);  // of 2^-52
    const int i1 = __float_as_int(m1) - 0x3BC00000, i2 = __float_as_int(m2) - 0x31400000;
    int64_t E = ((int64_t)thi << 32 | tlo) + ((int64_t)i1 << 21) + i2;
    constexpr int64_t one = 0x3FF0000000000000ll;
    if (E < one) E += E - one;  // below 1 the units are half as large (only from T = 1)
    if (!TAIL) return n < -1021 * kTab ? 0.0 : __longlong_as_double(E + ((int64_t)(n >> 9) << 52));
    if (n < -1021 * kTab) {  // below the normal range: the one rounding is the product's
        const double v = __longlong_as_double(E + ((int64_t)((n >> 9) + 64) << 52)) * 0x1p-64;
        return n < -1076 * kTab ? 0.0 : v;
    }
    return __longlong_as_double(E + ((int64_t)(n >> 9) << 52));
}

}  // namespace p64
}  // namespace tagi
