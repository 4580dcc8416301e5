// Extended floats on the integer pipes.
//
// GB300 issues one FP64 warp instruction per 64 cycles and SM sub-partition, a 32 x 32 -> 64 bit integer
// multiply-add (IMAD.WIDE) every 2 (measured: 2.2 against 67 cycles), so a chain of FP64 products costs less as
// integer products of 62-bit significands.  An xf holds a positive value m 2^e with m in [2^62, 2^63)
// ("normalised"; the functions say where slightly less is allowed).  A product keeps the upper 64 of 126 bits and drops
// the low partial product: relative error below 2^-59, 64 times smaller than an FP64 rounding.  Exponents are
// 32-bit integers, so nothing over- or underflows before the conversion to FP64.
// Signs are kept apart (a sign bit in bit 31 of a word), sums of signed terms stay in FP64.
//
// Host and device: the host builds the per-primitive records and the tables, and the CPU tests run the same code.
#pragma once

#include <cstdint>
#include <cstring>

#ifdef __CUDACC__
#define SHG_HD __host__ __device__ __forceinline__
// A translation unit whose loop bodies outgrow the instruction cache defines SHG_XF_CALLS: the longer functions are
// called instead of inlined (five operators in one pass, 200,000 pairs: 814 inlined, 752 us called; 1/r and erfc alone,
// 1M pairs: 2.49 inlined, 2.97 ms called)
#ifdef SHG_XF_CALLS
#define SHG_XF_LONG static __host__ __device__ __noinline__
#else
#define SHG_XF_LONG SHG_HD
#endif
#else
#define SHG_XF_LONG inline
#include <cmath>
#define SHG_HD inline
#endif

namespace shg {
namespace xfp {

struct xf {
    uint64_t m;
    int e;
};

SHG_HD uint64_t join(uint32_t hi, uint32_t lo) { return ((uint64_t)hi << 32) | lo; }
SHG_HD uint32_t hi32(uint64_t v) { return (uint32_t)(v >> 32); }
SHG_HD uint32_t lo32(uint64_t v) { return (uint32_t)v; }

// floor(a b / 2^64) - {0, 1, 2}: a < 2^63 and b < 2^63 (the two middle products then add up below 2^64)
SHG_HD uint64_t mulhi(uint64_t a, uint64_t b)
{
    uint64_t mid = (uint64_t)hi32(a) * lo32(b);
    mid += (uint64_t)lo32(a) * hi32(b);
    return (uint64_t)hi32(a) * hi32(b) + hi32(mid);
}

SHG_HD uint64_t dbits(double x)
{
#ifdef __CUDA_ARCH__
    return (uint64_t)__double_as_longlong(x);
#else
    uint64_t v;
    std::memcpy(&v, &x, sizeof v);
    return v;
#endif
}
SHG_HD double bitsd(uint64_t v)
{
#ifdef __CUDA_ARCH__
    return __longlong_as_double((long long)v);
#else
    double x;
    std::memcpy(&x, &v, sizeof x);
    return x;
#endif
}

SHG_HD uint32_t fbits(float x)
{
#ifdef __CUDA_ARCH__
    return __float_as_uint(x);
#else
    uint32_t v;
    std::memcpy(&v, &x, sizeof v);
    return v;
#endif
}

// product of two normalised xf: the raw significand is in [2^60, 2^62); one shift by 1 or 2 normalises it
SHG_HD xf mul(xf a, xf b)
{
    const uint64_t r = mulhi(a.m, b.m);
    const int s = 2 - (int)((hi32(r) >> 29) & 1u);
    return xf{r << s, a.e + b.e + 64 - s};
}

// raw product of two normalised xf: significand in [2^60, 2^62), for one further product by muln
SHG_HD xf mulr(xf a, xf b) { return xf{mulhi(a.m, b.m), a.e + b.e + 64}; }

SHG_HD int clz32(uint32_t v)
{
#ifdef __CUDA_ARCH__
    return __clz((int)v);
#else
    return __builtin_clz(v);
#endif
}

// normalised product where one factor may be raw (significand at least 2^60; error below 2^-57)
SHG_HD xf muln(xf a, xf b)
{
    const uint64_t r = mulhi(a.m, b.m);
    const int s = clz32(hi32(r)) - 1;
    return xf{r << s, a.e + b.e + 64 - s};
}

// v >> s, 0 for s > 63 (s >= 0)
SHG_HD uint64_t shr(uint64_t v, int s)
{
#ifdef __CUDA_ARCH__
    uint64_t r;
    asm("shr.b64 %0, %1, %2;" : "=l"(r) : "l"(v), "r"(s));
    return r;
#else
    return s > 63 ? 0 : v >> s;
#endif
}

// x^n, n >= 1
SHG_HD xf powi(xf x, int n)
{
    xf r = x;
#pragma unroll 1
    for (int i = 1; i < n; ++i) r = mul(r, x);
    return r;
}

// sum of two normalised xf (significands truncated at the larger exponent)
SHG_HD xf add(xf a, xf b)
{
    const int e = a.e > b.e ? a.e : b.e;
    const uint64_t m = shr(a.m, e - a.e) + shr(b.m, e - b.e);                // < 2^64
    const int c = (int)(hi32(m) >> 31);
    return xf{m >> c, e + c};
}

// positive normal FP64 value (exact); 0 and denormals give a value below 2^-1021
SHG_HD xf from_double(double x)
{
    const uint64_t v = dbits(x);
    const uint64_t m = ((v & 0xfffffffffffffull) | 0x10000000000000ull) << 10;
    return xf{m, (int)((uint32_t)(v >> 52) & 0x7ffu) - 1085};
}

// FP64 value with the sign of bit 31 of `sign`: round to nearest (ties up) of the 62-bit significand;
// below the normal range 0, above it infinity.  a.m in [2^62, 2^63).  Denormal results would take a shift by a variable
// count: five operators on 200,000 pairs 749 -> 765 us, 1/r and erfc on 1M pairs 2.489 -> 2.506 ms, 900,000 (a b a~) triples
// 11.36 -> 11.53 ms; in a branch of their own 790 us and 2.506 ms.
SHG_HD double to_double(xf a, uint32_t sign)
{
    const uint64_t r = (a.m + 512u) >> 10;                                   // 2^52 .. 2^53
    const int E = a.e + 1084;                                                // biased exponent less the implicit bit
    uint64_t v = r + ((uint64_t)(uint32_t)E << 52);
    if ((unsigned)E >= 2046u) v = E < 0 ? 0 : 0x7ff0000000000000ull;
    return bitsd(v | ((uint64_t)(sign & 0x80000000u) << 32));
}

#ifdef __CUDACC__
__device__ __forceinline__ float seed_rsqrt(float x)
{
    float r;
    asm("rsqrt.approx.f32 %0, %1;" : "=f"(r) : "f"(x));
    return r;
}
#endif

// 24-bit fraction y0 2^24 of the seed y0 2^-14 of 1 / sqrt(f), f in [1, 4): y0 in [1/2, 1).  Read off the float's bits as
// an offset from those of 2^-15, not as its mantissa: the approximation may fall an ulp or two short of 2^-15 for f just
// below 4 (its error bound is 2^-22.9), and the mantissa of such a float stands for almost twice its value.  Below 2^-15 the
// offset counts half units, so it gives at most 2^-25 less than the float per ulp: within the step's range.
SHG_HD uint32_t seed_fraction(float r)
{
    r = fminf(r, 6.1035152e-05f);                                            // the float below 2^-14
    return fbits(r) - (0x38000000u - 0x800000u);
}

// y0 (1 + h) 2^-h2 = 1 / sqrt(f 2^(2 h2)), f = M 2^-61 in [1, 4), from its seed, in fixed point: h = e/2 + 3 e^2/8,
// e = 1 - f y0^2 (|e| < 2^-20.5, two ulps of the seed; the dropped 5 e^3/16 is then 2^-63)
SHG_HD xf rsqrt_step(uint64_t M, int h2, uint32_t Y0)
{
    const uint64_t S = ((uint64_t)Y0 * Y0) << 15;                            // y0^2 2^63
    const int64_t e = (int64_t)((1ull << 60) - mulhi(M, S)) - 1;             // units 2^-60, |e| < 2^39.5
    const int32_t es = (int32_t)(e >> 9);
    const int32_t e2 = (int32_t)(((int64_t)es * es) >> 32);                  // units 2^-70
    const int64_t h = (e >> 1) + ((e2 * 3) >> 13);
    const uint64_t t1 = (uint64_t)Y0 * lo32((uint64_t)h);
    const int32_t t2 = (int32_t)Y0 * (int32_t)(h >> 32);
    const int64_t yh = (int64_t)(t1 + ((uint64_t)(uint32_t)t2 << 32)) >> 21; // y0 h, units 2^-63
    uint64_t Y = ((uint64_t)(Y0 << 7) << 32) + (uint64_t)yh;
    if (Y >> 63) Y = 0x7fffffffffffffffull;                                  // y = 1
    return xf{Y, -63 - h2};
}

// 1 / sqrt(a), a normalised: FP32 seed (2^-22) and one step of third order
SHG_XF_LONG xf rsqrt(xf a)
{
    const int odd = (a.e + 61) & 1;                                          // 1: shift the significand down once
    const uint64_t M = a.m >> odd;
    // the seed from the upper word f 2^29
    const float x = (float)hi32(M) * 0.5f;
#ifdef __CUDA_ARCH__
    const float r = seed_rsqrt(x);
#else
    const float r = (float)(1.0 / std::sqrt((double)x));
#endif
    return rsqrt_step(M, (a.e + 61 + odd) >> 1, seed_fraction(r));
}

// ------------------------------------------------------------------------- //
// exp(y) - 1 = y (1 + y/2 + y^2/6 + y^3/24 + y^4/120), 0 <= y <= 2^-9, with y = Y 2^-64 and the result in      //
// units 2^-63 (the dropped y^6/720 is below 2^-63).                                                             //
// ------------------------------------------------------------------------- //
SHG_HD uint64_t expm1_small(uint64_t Y)
{
    const uint32_t y = (uint32_t)(Y >> 23);                                  // y 2^41
    const uint32_t p4 = 178956971u + (uint32_t)(((uint64_t)y * 35791394u) >> 41);        // (1/24 + y/120) 2^32
    const uint32_t p3 = 715827883u + (uint32_t)(((uint64_t)y * p4) >> 41);               // 1/6 + ..., units 2^-32
    const uint64_t p2 = 0x4000000000000000ull + (((uint64_t)y * p3) >> 10);              // 1/2 + ..., units 2^-63
    const uint64_t p1 = 0x8000000000000000ull + mulhi(Y, p2);                            // 1 + ..., units 2^-63
    // Y (2^-64) times p1 (2^-63): p1 reaches 2^63, so halve it
    return mulhi(Y, p1 >> 1) << 1;
}

}  // namespace xfp
}  // namespace shg
