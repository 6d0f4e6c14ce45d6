// Rounding to bfloat16 (8 significant bits, ties to even) shared by the
// warm-start kernels.
#pragma once

#include <cuda_runtime.h>
#include <stdint.h>

namespace tagi {

// Nearest bfloat16 of a float64: the mantissa cut to 7 bits with the tie to
// even, as integers (float64 arithmetic runs at 1/73 of the float32 rate, and
// every CTA rounds the network's weights when it starts).  Below float32's
// normal range the spacing is 2^-133: scaled, rounded and scaled back there.
__device__ __forceinline__ uint16_t bf16_of_double(double x)
{
    const uint64_t b = (uint64_t)__double_as_longlong(x);
    const uint16_t sign = (uint16_t)((b >> 48) & 0x8000u);
    const int e = (int)((b >> 52) & 0x7ff) - 896;  // exponent field of float32
    if (e >= 1 && e <= 254) {
        const uint64_t m = (b & 0x7fffffffffffffffull) - (896ull << 52);
        return sign | (uint16_t)((m + 0xfffffffffffull + ((m >> 45) & 1)) >> 45);
    }
    if (isnan(x)) return 0x7FC0;
    if (e > 254) return sign | 0x7F80;
    return sign | (uint16_t)(__float_as_uint((float)(rint(fabs(x) * 0x1p133) * 0x1p-133)) >> 16);
}

__device__ __forceinline__ float bf16_float(uint32_t b) { return __uint_as_float(b << 16); }

// two float32 to bfloat16, `lo` in the low half
__device__ __forceinline__ uint32_t bf16x2(float lo, float hi)
{
    uint32_t r;
    asm("cvt.rn.bf16x2.f32 %0, %1, %2;" : "=r"(r) : "f"(hi), "f"(lo));
    return r;
}

}  // namespace tagi
