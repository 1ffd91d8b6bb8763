// fp64_int.cuh -- FP64 reciprocal and reciprocal square root refined on the
// integer pipe.
//
// GB300 has two FP64 lanes per SM and clock (1.6 measured with a chain of
// DFMAs) beside 60 to 107 integer lanes, and a kernel bound by its FP64 pipe
// leaves the integer pipe idle: 48 integer instructions beside each DFMA cost
// no DFMA throughput (measured).  The Newton-Raphson corrections of a
// reciprocal only touch the mantissa, so they need no alignment or
// normalisation: a handful of 32 x 32 -> 64-bit products replaces the four
// FP64 instructions of the reciprocal and the eight or so of CUDA's rsqrt.
//
// Both take the hardware's seed (rcp.approx.ftz.f64 / rsqrt.approx.ftz.f64:
// 21 mantissa bits, the low 32 bits of the result zero), form its residual e
// exactly enough in 64-bit fixed point, and apply the series to second order:
//   1/b     = y (1 + e + e^2 + ...),            e = 1 - b y
//   1/sqrtx = y (1 + e/2 + 3 e^2/8 + ...),      e = 1 - x y^2
// with |e| <= 2^-18.9, so what is left out is below 2^-56; the sum is rounded
// to nearest once: at most 0.53 ulp (reciprocal) and 0.57 ulp (square root)
// with seeds off by 2^-20 (the FP64 Newton form: 1 ulp and more).
#pragma once

#include <cstdint>

#include <cuda_runtime.h>

namespace hydro {

__host__ __device__ __forceinline__ uint32_t umulhi32(uint32_t a, uint32_t b)
{
    return static_cast<uint32_t>((static_cast<uint64_t>(a) * b) >> 32);
}

// The seed as a 21-bit mantissa (with the leading one) in the binade of the
// exact result, base: the word below that binade (exponent field - 1).  A
// seed rounded across the binade's end is clamped to it, so the product with
// the argument always has the same scale.
__host__ __device__ __forceinline__ uint32_t seed_mantissa(uint32_t yh, uint32_t base)
{
    const uint32_t lo = base + 0x100000u, hi = base + 0x1fffffu;
    yh &= 0x7fffffffu;
    yh = yh > lo ? yh : lo;
    yh = yh < hi ? yh : hi;
    return yh - base;
}

// Bits of 1/b for normal b with a normal reciprocal; yh: the seed's high word.
__host__ __device__ __forceinline__ uint64_t rcp_bits(uint64_t b, uint32_t yh)
{
    const uint32_t bl = static_cast<uint32_t>(b), bw = static_cast<uint32_t>(b >> 32);
    const uint32_t bh = (bw & 0xfffffu) | 0x100000u;
    const uint32_t base = 0x7fc00000u - (bw & 0x7ff00000u);
    const uint32_t my = seed_mantissa(yh, base);
    // mantissa product: 2^73 (1 - e); 2^73 vanishes modulo 2^64
    const uint64_t p = static_cast<uint64_t>(bl) * my + (static_cast<uint64_t>(bh * my) << 32);
    const int64_t e = -static_cast<int64_t>(p);                    // e 2^73, |e| < 2^-18
    const int32_t eh = static_cast<int32_t>(e >> 24);
    const uint32_t e2 = umulhi32(eh < 0 ? -eh : eh, eh < 0 ? -eh : eh);   // e^2 2^73 / 2^7
    const int64_t t = e + static_cast<int64_t>(static_cast<uint64_t>(e2) * 128u);
    const uint64_t r = ((static_cast<uint64_t>(my) << 42) | 512u)
                     + static_cast<uint64_t>(static_cast<int64_t>(static_cast<int32_t>(2 * my)) * static_cast<int32_t>(t >> 32))
                     + umulhi32(2 * my, static_cast<uint32_t>(t));
    return (r >> 10) + (static_cast<uint64_t>(base | (bw & 0x80000000u)) << 32);
}

// 1/sqrt(x) of normal positive x as a mantissa scaled 2^62, to 2^-59, and the
// word below its binade; yh: the seed's high word.
__host__ __device__ __forceinline__ uint64_t rsqrt_mantissa(uint64_t x, uint32_t yh, uint32_t &base)
{
    const uint32_t xl = static_cast<uint32_t>(x), xw = static_cast<uint32_t>(x >> 32);
    const uint32_t xh = (xw & 0xfffffu) | 0x100000u;
    base = 0x5fd00000u - (((xw + 0x100000u) >> 1) & 0x7ff00000u);
    const uint32_t my = seed_mantissa(yh, base);
    // odd powers of two: double one factor, so that x y^2 = 2^94 (1 - e)
    const uint32_t odd = (~xw >> 20) & 1u;
    const uint64_t m2 = static_cast<uint64_t>(my) * (my << odd);
    const uint32_t m0 = static_cast<uint32_t>(m2), m1 = static_cast<uint32_t>(m2 >> 32);
    const uint64_t s = static_cast<uint64_t>(xh) * m0 + umulhi32(xl, m0) + static_cast<uint64_t>(xl) * m1
                     + (static_cast<uint64_t>(xh * m1) << 32);     // (x y^2) 2^62
    const int64_t e = static_cast<int64_t>((1ull << 62) - s);      // e 2^62, |e| < 2^-17
    const int32_t eh = static_cast<int32_t>(e >> 14);
    const uint32_t e2 = umulhi32(eh < 0 ? -eh : eh, eh < 0 ? -eh : eh);   // 4 e^2 2^62
    // e/2 + 3 e^2/8, scaled 2^74
    const int64_t t = static_cast<int64_t>(static_cast<uint64_t>(e) << 11)
                    + static_cast<int64_t>(static_cast<uint64_t>(e2) * 384u);
    return (static_cast<uint64_t>(my) << 42)
         + static_cast<uint64_t>(static_cast<int64_t>(static_cast<int32_t>(my)) * static_cast<int32_t>(t >> 32))
         + umulhi32(my, static_cast<uint32_t>(t));
}

// Bits of 1/sqrt(x) for normal positive x.
__host__ __device__ __forceinline__ uint64_t rsqrt_bits(uint64_t x, uint32_t yh)
{
    uint32_t base;
    const uint64_t r = rsqrt_mantissa(x, yh, base) + 512u;
    return (r >> 10) + (static_cast<uint64_t>(base) << 32);
}

// Bits of k / sqrt(x) for normal positive x and k (bits kb), rounded once: the
// factor joins before the rounding, a 64 x 64-bit product's upper half (the
// lowest partial product, below 2^-61, left out).
__host__ __device__ __forceinline__ uint64_t rsqrt_scaled_bits(uint64_t x, uint32_t yh, uint64_t kb)
{
    uint32_t base;
    const uint64_t r = rsqrt_mantissa(x, yh, base);
    const uint32_t rh = static_cast<uint32_t>(r >> 32), rl = static_cast<uint32_t>(r);
    const uint32_t kh = (static_cast<uint32_t>(kb >> 21) & 0x7fffffffu) | 0x80000000u, kl = static_cast<uint32_t>(kb) << 11;
    uint64_t p = static_cast<uint64_t>(rh) * kh + umulhi32(rh, kl) + umulhi32(rl, kh);   // product of the mantissas, 2^61
    const bool two = (p >> 62) != 0;                                                   // 2 <= product < 4
    p = (two ? p : p << 1) + 512u;
    const uint32_t e = base + (static_cast<uint32_t>(kb >> 32) & 0x7ff00000u) - 0x3ff00000u + (two ? 0x100000u : 0u);
    return (p >> 10) + (static_cast<uint64_t>(e) << 32);
}

}  // namespace hydro
