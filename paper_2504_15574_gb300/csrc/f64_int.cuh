// f64_int.cuh -- FP64 products on the integer pipe, for the FP64 path of stage_f64.cu.
//
// GB300 issues one FP64 warp instruction per 64 cycles and scheduler (2 FP64 lanes per SM); a product
// rounded to nearest even takes about 40 integer instructions, which issue beside the FP64 pipe's
// work.  Each function returns the IEEE product (round to nearest even; a zero product is +0), given
// that its operands are normal (or zero where it says so) and its product is normal: callers bound
// the exponents of what they load (f64_within) and take plain forms outside.  Plain C++ but for the
// qualifiers, so that the same code is checked on the host against the hardware's products.
#pragma once

#include <math.h>
#include <stdint.h>
#include <string.h>

#if defined(__CUDACC__)
#define F64I __host__ __device__ __forceinline__
#else
#define F64I static inline
#endif

namespace vk {

F64I uint64_t f64_bits(double x)
{
#if defined(__CUDA_ARCH__)
    return (uint64_t)__double_as_longlong(x);
#else
    uint64_t u;
    memcpy(&u, &x, 8);
    return u;
#endif
}

// The two words of x.  On the device behind an inline move: the compiler turns a zero test on the bits of
// a double that it can see back into a comparison on the FP64 pipe.
F64I void f64_split(double x, uint32_t &hi, uint32_t &lo)
{
#if defined(__CUDA_ARCH__)
    asm("mov.b64 {%0, %1}, %2;" : "=r"(lo), "=r"(hi) : "d"(x));
#else
    const uint64_t u = f64_bits(x);
    hi = (uint32_t)(u >> 32);
    lo = (uint32_t)u;
#endif
}

F64I bool f64_zero(double x)
{
    uint32_t hi, lo;
    f64_split(x, hi, lo);
    return ((hi << 1) | lo) == 0;
}

F64I double f64_of(uint32_t hi, uint32_t lo)
{
#if defined(__CUDA_ARCH__)
    return __hiloint2double((int)hi, (int)lo);
#else
    const uint64_t u = ((uint64_t)hi << 32) | lo;
    double x;
    memcpy(&x, &u, 8);
    return x;
#endif
}

// x is zero, or |x| in [2^-lo, 2^hi)
template <int LO, int HI>
F64I bool f64_within(double x)
{
    uint32_t hi, lo;
    f64_split(x, hi, lo);
    return ((hi << 1) | lo) == 0 || ((hi >> 20) & 0x7ffu) - (uint32_t)(1023 - LO) < (uint32_t)(LO + HI);
}

// x 2^K, |K| <= 4; x may be zero
template <int K>
F64I double scale2(double x)
{
    uint32_t hi, lo;
    f64_split(x, hi, lo);
    return f64_of(((hi << 1) | lo) == 0 ? hi : hi + (uint32_t)(K * (1 << 20)), lo);
}

// a b, neither zero.  The 106-bit product of the two 53-bit significands from four 32-bit products;
// its leading 53 bits (n = 1: the significands' product is 2 or more) plus the rounding increment, whose
// carry out of the significand raises the exponent by itself.
F64I double mul_int(double a, double b)
{
    uint32_t ah, al, bh, bl;
    f64_split(a, ah, al);
    f64_split(b, bh, bl);
    const uint32_t am = (ah & 0xfffffu) | 0x100000u, bm = (bh & 0xfffffu) | 0x100000u;
    const uint64_t ll = (uint64_t)al * bl;
    const uint64_t mid = (uint64_t)am * bl + ((uint64_t)al * bm + (ll >> 32));
    const uint64_t top = (uint64_t)am * bm + (mid >> 32);   // product / 2^64, in [2^40, 2^42)
    const uint32_t n = (uint32_t)(top >> 41), sh = 20u + n, ml = (uint32_t)mid;
    const uint32_t m0 = (uint32_t)(((((uint64_t)(uint32_t)top) << 32) | ml) >> sh);
    const uint32_t m1 = (uint32_t)(top >> sh);
    const uint32_t rest = (ml << (32u - sh)) | ((uint32_t)ll != 0u ? 1u : 0u);   // dropped bits, sticky last
    const uint32_t inc = rest + (m0 & 1u) > 0x80000000u ? 1u : 0u;
    // exponent sum - 1023 + n - 1 (the significand's leading bit adds one), modulo 2^32 above the sign
    const uint32_t ef = (ah & 0x7ff00000u) + (bh & 0x7ff00000u) - (1024u << 20) + (n << 20);
    const uint64_t m = (((uint64_t)m1 << 32) | m0) + inc;
    return f64_of(((uint32_t)(m >> 32) + ef) | ((ah ^ bh) & 0x80000000u), (uint32_t)m);
}

// a b where a may be zero
F64I double mul_int_z(double a, double b)
{
    const double p = mul_int(a, b);
    return f64_zero(a) ? 0.0 : p;
}

// a b where either may be zero
F64I double mul_int_zz(double a, double b)
{
    const double p = mul_int(a, b);
    return f64_zero(a) || f64_zero(b) ? 0.0 : p;
}

// a^2, a may be zero
F64I double sq_int(double a) { return mul_int_z(a, a); }

// a + b, neither negative, either may be zero.  The smaller significand is shifted right to the larger's
// exponent, with ten spare bits below (what falls out of them only sets the last one), added, and
// rounded as in mul_int; shifts of 64 bits and more leave the larger value as it is.
F64I double add_pos(double a, double b)
{
    uint32_t ah, al, bh, bl;
    f64_split(a, ah, al);
    f64_split(b, bh, bl);
    const bool less = ah < bh;   // (equal high words have the same exponent: either order will do)
    const uint32_t xh = less ? bh : ah, xl = less ? bl : al, yh = less ? ah : bh, yl = less ? al : bl;
    const uint32_t d = (xh >> 20) - (yh >> 20);
    // significands above ten spare bits: [2^62, 2^63), zero for a zero
    const uint64_t x = (((uint64_t)((xh & 0xfffffu) | 0x100000u) << 32) | xl) << 10;
    const uint64_t y0 = (((uint64_t)((yh & 0xfffffu) | 0x100000u) << 32) | yl) << 10;
    const uint64_t y = (d > 63u || (yh | yl) == 0) ? 0 : y0 >> d;
    const uint64_t lost = (d > 63u || d == 0u || (yh | yl) == 0) ? 0 : y0 << (64u - d);
    const uint64_t sum = x + y;
    const uint32_t n = (uint32_t)(sum >> 63), sh = 10u + n;
    const uint64_t m = sum >> sh;
    const uint32_t rest = ((uint32_t)sum << (32u - sh)) | (lost != 0 ? 1u : 0u);
    const uint32_t inc = rest + ((uint32_t)m & 1u) > 0x80000000u ? 1u : 0u;
    const uint64_t r = m + inc;
    const uint32_t h = (uint32_t)(r >> 32) + (xh & 0x7ff00000u) - 0x100000u + (n << 20);
    const bool zero = (xh | xl) == 0;
    return f64_of(zero ? 0u : h, zero ? 0u : (uint32_t)r);
}

// x N for a small odd N (3, 5, 7 or 11); x may be zero
template <int N>
F64I double mul_small(double x)
{
    uint32_t hi, lo;
    f64_split(x, hi, lo);
    const uint64_t p = ((((uint64_t)(hi & 0xfffffu)) << 32) | lo) * N + ((uint64_t)N << 52);
    constexpr int S0 = N >= 8 ? 3 : N >= 4 ? 2 : 1;   // p >> S0 has 53 or 54 bits
    const uint32_t n = (uint32_t)(p >> (53 + S0)), sh = S0 + n;
    const uint64_t m = p >> sh;
    const uint32_t rest = (uint32_t)p << (32u - sh);
    const uint32_t inc = rest + ((uint32_t)m & 1u) > 0x80000000u ? 1u : 0u;
    const uint64_t r = m + inc;
    const bool zero = ((hi << 1) | lo) == 0;
    const uint32_t h = ((uint32_t)(r >> 32) + ((hi & 0x7ff00000u) - 0x100000u) + (sh << 20)) | (hi & 0x80000000u);
    return f64_of(zero ? hi : h, zero ? lo : (uint32_t)r);
}

// ---- division by a constant -----------------------------------------------------------
// 1/d as h + l, h = 1/d rounded toward zero, l > 0 the remainder: x / d is RN(x h + RN(x l)), a product
// and one fused operation.  d itself serves the plain forms, which divide (1/d need not be a normal number there).
struct DivC { double h, l, d; };

// Where 1/d is a double, l = h 2^-120: x h is then exact and what l adds is far below half its ulp, while
// x l stays a normal number for the x of the integer form (a subnormal l is no operand of mul_int); a
// positive l also keeps an infinite x infinite.
inline DivC div_const_of(double d)
{
    double y = 1.0 / d, r = fma(-y, d, 1.0);
    if (r < 0.0) {
        y = nextafter(y, 0.0);
        r = fma(-y, d, 1.0);
    }
    const double l = r > 0.0 ? r / d : y * 0x1p-120;
    return DivC{y, l > 0.0 ? l : 4.9406564584124654e-324, d};
}

F64I double fma_rn(double a, double b, double c)
{
#if defined(__CUDA_ARCH__)
    return __fma_rn(a, b, c);
#else
    return fma(a, b, c);
#endif
}

// x / d with the product by l on the integer pipe; x zero or well inside the normal range.
F64I double div_const_int(double x, const DivC &d) { return fma_rn(x, d.h, mul_int_z(x, d.l)); }

}  // namespace vk
