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

#include <initializer_list>

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

F64I uint32_t f64_hi(double x)
{
#if defined(__CUDA_ARCH__)
    return (uint32_t)__double2hiint(x);
#else
    return (uint32_t)(f64_bits(x) >> 32);
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

F64I double fma_rn(double a, double b, double c)
{
#if defined(__CUDA_ARCH__)
    return __fma_rn(a, b, c);
#else
    return fma(a, b, c);
#endif
}

// ---- division by a constant -----------------------------------------------------------
// 1/d as h + l, h = 1/d rounded toward zero, l > 0 the remainder: x / d is RN(x h + RN(x l)), a product
// and one fused operation (Brisebarre and Muller, "Correctly rounded multiplication by arbitrary precision
// constants", 2005).  d itself is for the plain forms, which divide (1/d need not be a normal number there).
struct DivC { double h, l, d; };

F64I double div_const(double x, const DivC &d) { return fma_rn(x, d.h, x * d.l); }

// The same with the product by l on the integer pipe; x zero or well inside the normal range.
F64I double div_const_int(double x, const DivC &d) { return fma_rn(x, d.h, mul_int_z(x, d.l)); }

// Whether c gives the rounded quotient x / d for every x.  The value before its last rounding is within
// 2^-103 of x / d, relatively, so only an x whose quotient is that near to a rounding boundary can miss.
// With the integer significands X and D the boundaries are odd N over 2^53 (X >= D) or 2^54 (X < D), and
// |X 2^k - N D| = |c| of such an x is below 2^-103 N D < 16: the x are found by solving N D = -c mod 2^k for
// every small c (at most a few dozen) and tried.
inline bool div_const_exact(const DivC &c)
{
    int e;
    uint64_t D = (uint64_t)ldexp(frexp(c.d, &e), 53);
    int t = 0;
    for (; !(D & 1); D >>= 1) ++t;   // c.d = D 2^t, D odd: 2^t divides every c
    uint64_t inv = D;                // D^-1 mod 2^64
    for (int k = 0; k < 6; ++k) inv *= 2 - D * inv;
    for (int k = 53; k <= 54; ++k)
        for (int64_t r = -(16 >> t); t <= 4 && r <= (16 >> t); ++r) {
            const uint64_t mod = 1ull << (k - t), n0 = (0 - (uint64_t)r * inv) & (mod - 1);
            for (uint64_t N = n0; N < (1ull << 54); N += mod) {
                if (N < (1ull << 53) || !(N & 1)) continue;
                const uint64_t X = (uint64_t)(((__int128)N * (int64_t)D + r) >> (k - t));
                if (X < (1ull << 52) || X >= (1ull << 53) || (X >= D << t) != (k == 53)) continue;
                const double x = (double)X;
                if (div_const(x, c) != x / c.d) return false;
            }
        }
    return true;
}

// The constant of a divisor d.  Where 1/d is a double, l = h 2^-120: x h is then exact and what l adds is far
// below half its ulp, while x l stays a normal number for the x of the integer form (a subnormal l is no
// operand of mul_int); a positive l also keeps an infinite x infinite.  Otherwise l is the rounded remainder,
// or a neighbour of it where some quotient would be missed with that one (every quotient is then the rounded
// one for all but 1.8 % of divisors, and for those all but one or two significands x).
inline DivC div_const_of(double d)
{
    double y = 1.0 / d, r = fma(-y, d, 1.0);
    if (r < 0.0) {
        y = nextafter(y, 0.0);
        r = fma(-y, d, 1.0);
    }
    const double l = r > 0.0 ? r / d : y * 0x1p-120;
    const DivC c{y, l > 0.0 ? l : 4.9406564584124654e-324, d};
    if (r > 0.0 && fabs(d) > 0x1p-500 && fabs(d) < 0x1p500)
        for (double v : {l, nextafter(l, 1.0), nextafter(l, 0.0)})
            if (div_const_exact(DivC{y, v, d})) return DivC{y, v, d};
    return c;
}

// ---- division -------------------------------------------------------------------------
// 1 / b to 2^-44 for a positive b in [2^-500, 2^500]: the leading 24 bits of b's significand through
// the hardware's FP32 reciprocal, one error term with the remaining bits, assembled into a double by
// integer operations.
F64I double recip_seed(double b)
{
#if defined(__CUDA_ARCH__)
    const int hi = __double2hiint(b), lo = __double2loint(b);
    const float bh = __int_as_float(0x3f800000 | ((hi & 0xfffff) << 3) | (int)((unsigned)lo >> 29));
    float r0;
    asm("rcp.approx.ftz.f32 %0, %1;" : "=f"(r0) : "f"(bh));
#else
    const uint64_t b64 = f64_bits(b);
    const int hi = (int)(b64 >> 32), lo = (int)(uint32_t)b64, hb = 0x3f800000 | ((hi & 0xfffff) << 3) | (int)((unsigned)lo >> 29);
    float bh;
    memcpy(&bh, &hb, 4);
    float r0 = 1.0f / bh;
#endif
    const float bl = (float)(lo & 0x1fffffff) * 0x1p-52f;
    r0 = fmaxf(fminf(r0, 0.99999994f), 0.5f);   // inside one binade: the error term is added to its bits
    float e = fmaf(-bh, r0, 1.0f);
    e = fmaf(-bl, r0, e);
#if defined(__CUDA_ARCH__)
    const float r1 = __fmul_rn(r0, __fmaf_rn(e, e, e));
    const int u = __float_as_int(r0), i1 = __float2int_rn(__fmul_rn(r1, 0x1p53f));
    long long bits = ((long long)((u >> 3) + ((1023 - 127) << 20)) << 32) | (unsigned)(u << 29);
    bits += i1;
    bits -= (long long)((hi >> 20) - 1023) << 52;
    return __longlong_as_double(bits);
#else
    const float r1 = r0 * fmaf(e, e, e);
    int u;
    memcpy(&u, &r0, 4);
    int64_t bits = (int64_t)((uint64_t)((u >> 3) + ((1023 - 127) << 20)) << 32 | (uint32_t)((uint32_t)u << 29));
    bits += lrintf(r1 * 0x1p53f);
    bits -= (int64_t)((hi >> 20) - 1023) * ((int64_t)1 << 52);
    return f64_of((uint32_t)((uint64_t)bits >> 32), (uint32_t)(uint64_t)bits);
#endif
}

// Whether q, within an ulp or two of a / b, is surely the rounded quotient (b positive): the remainder
// a - b q, which one fused operation gives exactly, is below half an ulp of q times b.  Only the high words
// are compared (a false alarm in 2^20).  256 x 512: 1,405 us a step, 1,359 without any check, 1,530 with the
// remainder from the integer significands (20 integer operations more instead of one FP64 operation).  Below a power of two the boundary is a quarter of an ulp away, but no quotient of two doubles is between
// there and q.
F64I bool quotient_rounded(double a, double b, double q)
{
    const uint32_t r = f64_hi(fma_rn(-b, q, a)) & 0x7fffffffu;
    return r < f64_hi(b) + (f64_hi(q) & 0x7ff00000u) - (1076u << 20);
}

// a / b for such a b: the product with the seed on the integer pipe (a zero or well inside the normal
// range), then one residual correction in two FP64 operations (Markstein 1990).  The corrected value is
// within 2^-88 of a / b before its rounding, which one quotient in about 2^35 does not survive: miss is set
// for it, and the caller divides.
F64I double div_pos(double a, double b, bool &miss)
{
    const double r = recip_seed(b), q0 = mul_int_z(a, r);
    const double q = fma_rn(fma_rn(-b, q0, a), r, q0);
    miss |= !quotient_rounded(a, b, q);
    return q;
}

}  // namespace vk
