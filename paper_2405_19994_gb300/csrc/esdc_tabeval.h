// One cubic of a table evaluated to FP64 accuracy without FP64 instructions.
//
// GB300 issues two FP64 lane operations per SM and clock, 64 times fewer than
// FP32's: an FP64 Horner step of a warp takes as long as about 70 FP32 or
// integer instructions of it.  A cubic on a narrow interval is its centre value
// plus a small bracket,
//   f(t) = c0 + B(t),  B(t) = t (c1 + t (c2 + t c3)),  |B| < 2^-8 S,
// S a power of two above |f| on the interval, so B needs 46 of f's 54 bits.  It
// is formed in pairs of FP32 numbers (error-free products by FMA, Knuth's
// two-sum; T. J. Dekker, Numer. Math. 18, 1971; D. E. Knuth, TAOCP 2, 4.2.2),
// scaled by 1/S, split at 2^-30 S and added to c0 as a 64-bit integer in units
// of 2^-57 S; the sum is then normalised and rounded to nearest by integer
// operations: 25 FP32 and about 25 integer instructions where Horner's rule
// took three FP64 ones.
//
// Error, in units of S: 2^-58 from c0's rounding, 2^-58 from the last part's,
// about 2^-46 |B|/S <= 2^-54 from the FP32 pairs (2^-56 at the usual |B| < 2^-10),
// and the final rounding to 53 bits, half an ulp of f: the tables' build checks
// compare this very function with long double.  Horner's rule rounded c0 and
// its last sum, half an ulp of f each.
//
// The same code runs on the host (the build checks); every FP32 operation is
// rounded by itself (no contraction) on both.
#pragma once
#include <cmath>
#include <cstdint>
#include <cstring>

#if defined(__CUDACC__)
#define ESDC_HD __host__ __device__ __forceinline__
#else
#define ESDC_HD inline
#endif

namespace esdc {

struct TabPoly {                    // 32 bytes
    int64_t c0;                     // 2^57 c0 / S
    float c1h, c1l, c2h, c2l, c3;   // c_k / S
    int32_t eS;                     // S = 2^eS
};

ESDC_HD float t_add(float a, float b)
{
#if defined(__CUDA_ARCH__)
    return __fadd_rn(a, b);
#else
    return a + b;
#endif
}
ESDC_HD float t_mul(float a, float b)
{
#if defined(__CUDA_ARCH__)
    return __fmul_rn(a, b);
#else
    return a * b;
#endif
}
ESDC_HD float t_fma(float a, float b, float c)
{
#if defined(__CUDA_ARCH__)
    return __fmaf_rn(a, b, c);
#else
    return std::fma(a, b, c);
#endif
}
ESDC_HD float t_float(uint32_t u)
{
#if defined(__CUDA_ARCH__)
    return __uint_as_float(u);
#else
    float f;
    std::memcpy(&f, &u, 4);
    return f;
#endif
}
ESDC_HD uint32_t t_bits(float f)
{
#if defined(__CUDA_ARCH__)
    return __float_as_uint(f);
#else
    uint32_t u;
    std::memcpy(&u, &f, 4);
    return u;
#endif
}
ESDC_HD int t_int(float f)          // round to nearest even
{
#if defined(__CUDA_ARCH__)
    return __float2int_rn(f);
#else
    return (int)std::nearbyint(f);
#endif
}

// t = th + tl: th the leading 24 bits (truncated), tl the other 29 rounded to 24;
// both 0 for |t| < 2^-73, which no bracket resolves.
ESDC_HD void tab_split(double t, float& th, float& tl)
{
    uint64_t b;
#if defined(__CUDA_ARCH__)
    b = (uint64_t)__double_as_longlong(t);
#else
    std::memcpy(&b, &t, 8);
#endif
    const uint32_t hi = (uint32_t)(b >> 32), lo = (uint32_t)b, ex = (hi >> 20) & 0x7ffu, sg = hi & 0x80000000u;
    th = tl = 0.0f;
    if (ex < 950u) return;
    th = t_float(sg | ((ex - 896u) << 23) | ((hi & 0xfffffu) << 3) | (lo >> 29));
    tl = t_mul((float)(int)(lo & 0x1fffffffu), t_float(sg | ((ex - 948u) << 23)));
}

ESDC_HD double tab_eval(const TabPoly& c, float th, float tl)
{
    // t c2 + t^2 c3: p1 + lo, lo below p1's last place (the quick two-sum: where c3's term
    // leads, what it drops is 2^-24 of that term)
    const float u = t_fma(th, c.c3, c.c2l);
    const float p0 = t_mul(th, c.c2h);
    const float l0 = t_fma(th, u, t_fma(tl, c.c2h, t_fma(th, c.c2h, -p0)));
    const float p1 = t_add(p0, l0);
    const float lo = t_add(l0, -t_add(p1, -p0));
    // c1 + that: sh + sl (Knuth's two-sum of the leading parts)
    const float sh = t_add(c.c1h, p1), bb = t_add(sh, -c.c1h);
    const float er = t_add(t_add(c.c1h, -t_add(sh, -bb)), t_add(p1, -bb));
    const float sl = t_add(er, t_add(c.c1l, lo));
    // B = t (sh + sl): P + L
    const float P = t_mul(th, sh);
    const float L = t_fma(th, sl, t_fma(tl, sh, t_fma(th, sh, -P)));
    // B in units of 2^-57: the part above 2^-30 from the sum with 1.5 2^-7 (whose last
    // place is 2^-30), the rest as an integer
    const float M = 1.5f / 128.0f;
    const float q = t_add(P, M);
    const float r = t_add(t_add(P, -t_add(q, -M)), L);
    const int i1 = (int)(t_bits(q) - t_bits(M));
    const int i2 = t_int(t_mul(r, 144115188075855872.0f));          // 2^57
    const int64_t v = c.c0 + ((int64_t)i1 * (1 << 27) + i2);
    // v 2^(eS - 57) as a double, rounded to nearest (ties away)
    const uint64_t a = v < 0 ? (uint64_t)(-v) : (uint64_t)v;
    if (a == 0) return 0.0;
#if defined(__CUDA_ARCH__)
    const int lz = __clzll((long long)a);
#else
    const int lz = __builtin_clzll(a);
#endif
    const uint64_t m = a << lz;
    const uint64_t bits = (((uint64_t)(1028 + c.eS - lz) << 52) + (m >> 11) + ((m >> 10) & 1u)) |
                          (v < 0 ? 0x8000000000000000ULL : 0ULL);
#if defined(__CUDA_ARCH__)
    return __longlong_as_double((long long)bits);
#else
    double d;
    std::memcpy(&d, &bits, 8);
    return d;
#endif
}

// Host: packs the cubic coef[0..3] (in t, |t| <= h); false if its scale leaves
// the exponent range that tab_eval composes.
inline bool tab_pack(const long double* coef, long double h, TabPoly& o)
{
    const long double br = h * (fabsl(coef[1]) + h * (fabsl(coef[2]) + h * fabsl(coef[3])));
    long double top = fabsl(coef[0]) + br;
    if (top < 260.0L * br) top = 260.0L * br;
    o = TabPoly{};
    if (!(top > 0.0L)) return top == 0.0L;                    // the zero function
    int e;
    frexpl(top, &e);                                          // top < 2^e
    if (e < -900 || e > 900) return false;
    o.eS = e;
    o.c0 = (int64_t)llrintl(ldexpl(coef[0], 57 - e));
    const long double c1 = ldexpl(coef[1], -e), c2 = ldexpl(coef[2], -e);
    o.c1h = (float)c1;
    o.c1l = (float)(c1 - (long double)o.c1h);
    o.c2h = (float)c2;
    o.c2l = (float)(c2 - (long double)o.c2h);
    o.c3 = (float)ldexpl(coef[3], -e);
    return std::isfinite(o.c1h) && std::isfinite(o.c2h) && std::isfinite(o.c3);
}

}  // namespace esdc
