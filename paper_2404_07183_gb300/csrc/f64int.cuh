// f64int.cuh -- float64 subtraction and multiplication on the integer pipes.
//
// GB300's float64 pipe takes one warp instruction per 65 to 77 cycles and SM
// sub-partition, whether its lanes are predicated on or off, so a float64 walk
// is bound by its float64 operations with most issue slots idle.  The
// functions here compute what the float64 instructions compute (round to
// nearest, ties to even: the same bits) from the mantissas as integers, in 40
// to 60 cycles of the integer pipes, which run beside the float64 one.  They
// hold for the operand ranges stated; the caller keeps others away from them.
#pragma once

#include <cstdint>

namespace pcfgb {

#ifdef __CUDACC__
#define PCF_HD __host__ __device__ __forceinline__
#else
#define PCF_HD inline
#endif

PCF_HD int f64i_clz(uint64_t x)
{
#ifdef __CUDA_ARCH__
    return __clzll((long long)x);
#else
    return x ? __builtin_clzll(x) : 64;
#endif
}

constexpr uint64_t kMant = (1ull << 52) - 1;
// Ends of a walk with biased exponents in this range and c >= n / 2^10 suit
// f64i_width: differences stay normal numbers (or 0).
constexpr uint32_t kWidthExpLo = 300, kWidthExpHi = 1700;
constexpr int kWidthOctaves = 10;

// The number with mantissa S (top bit 62, the bits below bit 10 to be rounded)
// and biased exponent e of that top bit.
PCF_HD uint64_t f64i_round(uint64_t S, uint32_t e)
{
    S += 0x1ff + ((S >> 10) & 1u);
    return (S >> 10) + ((uint64_t)(e - 1u) << 52);   // the top bit (or its carry) adds to e - 1
}

// n - c for bit patterns 0 < c <= n whose exponents differ by kWidthOctaves at
// most (no bit of c is lost when it is aligned to n), within the range above.
PCF_HD uint64_t f64i_width(uint64_t n, uint64_t c)
{
    const uint32_t en = (uint32_t)(n >> 52), ec = (uint32_t)(c >> 52);
    const uint64_t a = ((n & kMant) | (kMant + 1)) << 10;
    const uint64_t b = ((c & kMant) | (kMant + 1)) << 10;
    const uint64_t d = a - (b >> ((en - ec) & 31u));
    const int lz = f64i_clz(d);                      // 1 .. 64
    const uint64_t r = f64i_round(d << ((lz - 1) & 63), en + 1u - (uint32_t)lz);
    return d ? r : 0;
}

// a * b, sign included, for factors that are 0 or 2^-510 to 2^510 in magnitude
// (the product is a normal number).
PCF_HD uint64_t f64i_mul(uint64_t a, uint64_t b)
{
    const uint32_t ea = (uint32_t)(a >> 52) & 0x7ffu, eb = (uint32_t)(b >> 52) & 0x7ffu;
    const uint64_t x = ((a & kMant) | (kMant + 1)) << 11;     // top bit 63
    const uint64_t y = ((b & kMant) | (kMant + 1)) << 10;     // top bit 62
#ifdef __CUDA_ARCH__
    const uint64_t hi = __umul64hi(x, y);
#else
    const uint64_t hi = (uint64_t)(((unsigned __int128)x * y) >> 64);
#endif
    uint64_t p = hi | ((x * y) != 0 ? 1u : 0u);               // sticky; top bit 61 or 62
    uint32_t e = ea + eb - 1023u;                             // exponent of bit 61
    if (p >> 62) ++e; else p <<= 1;
    const uint64_t sign = (a ^ b) & (1ull << 63);
    return ea == 0u || eb == 0u ? sign : f64i_round(p, e) | sign;
}

// Values whose products and squared differences suit f64i_mul: 0, or 2^-400 to
// 2^500 in magnitude (a difference is then 0 or at least 2^-452).
PCF_HD bool f64i_value_suits(uint64_t v)
{
    const uint32_t e = (uint32_t)(v >> 52) & 0x7ffu;
    return (v << 1) == 0 || (e >= 623u && e <= 1523u);
}

}  // namespace pcfgb
