// psgld_normals.cuh -- packed FP32 arithmetic, and four standard normals from
// four random words in it.
//
// Compiles for the host too, where every operation rounds as on the device
// (multiply-adds, products, conversions and sqrtf are IEEE operations), so
// that a host program can evaluate the function at every argument.
#pragma once

#include <math.h>
#include <stdint.h>
#include <string.h>
#include <vector_functions.h>
#include <vector_types.h>

#ifdef __CUDACC__
#define PSGLD_HDI __host__ __device__ __forceinline__
#else
#define PSGLD_HDI inline
#endif

namespace psgld {
namespace dev {

PSGLD_HDI float as_float(uint32_t x)
{
#ifdef __CUDA_ARCH__
    return __uint_as_float(x);
#else
    float f;
    memcpy(&f, &x, sizeof f);
    return f;
#endif
}

PSGLD_HDI uint32_t as_bits(float x)
{
#ifdef __CUDA_ARCH__
    return __float_as_uint(x);
#else
    uint32_t u;
    memcpy(&u, &x, sizeof u);
    return u;
#endif
}

// Two FP32 operations per instruction (the sm_100 family's packed FP32
// arithmetic), each rounded like its scalar form.
PSGLD_HDI float2 fma2(float2 a, float2 b, float2 c)
{
#ifdef __CUDA_ARCH__
    float2 d;
    asm("fma.rn.f32x2 %0, %1, %2, %3;"
        : "=l"(reinterpret_cast<unsigned long long &>(d))
        : "l"(reinterpret_cast<unsigned long long &>(a)), "l"(reinterpret_cast<unsigned long long &>(b)),
          "l"(reinterpret_cast<unsigned long long &>(c)));
    return d;
#else
    return make_float2(fmaf(a.x, b.x, c.x), fmaf(a.y, b.y, c.y));
#endif
}

PSGLD_HDI float2 mul2(float2 a, float2 b)
{
#ifdef __CUDA_ARCH__
    float2 d;
    asm("mul.rn.f32x2 %0, %1, %2;"
        : "=l"(reinterpret_cast<unsigned long long &>(d))
        : "l"(reinterpret_cast<unsigned long long &>(a)), "l"(reinterpret_cast<unsigned long long &>(b)));
    return d;
#else
    return make_float2(a.x * b.x, a.y * b.y);
#endif
}

PSGLD_HDI float2 both(float x) { return make_float2(x, x); }

// Four normals from four random words: uniforms on (0, 1), u = the top 23
// bits plus one half, times 2^-23 (exact in FP32); Box and Muller's transform
// (Ann. Math. Statist. 29, 1958) of (u0, u1) and (u2, u3), cos first, then sin.
//
// Instructions bound every kernel that draws noise, so the two pairs go
// through packed arithmetic, and logarithm, sine and cosine are written for
// the arguments they meet here (no subnormals, no infinities, no large
// angles), after Cody and Waite, Software Manual for the Elementary Functions
// (1980): chapter 5's split of the logarithm's argument into exponent and a
// fraction in [sqrt(1/2), sqrt(2)), chapter 8's reduction of the angle to the
// nearest quarter turn, with minimax polynomials (Cheney, Introduction to
// Approximation Theory, 1966) found by linear programming on Chebyshev nodes:
//  * u0: the bits under the exponent of 1 give 1 + m 2^-23; subtracting
//    1 - 2^-24 is exact.
//  * -2 ln u0: u0 = 2^e (1 + g), g in [sqrt(1/2) - 1, sqrt(2) - 1];
//    -2 ln(1 + g) = h + h^2 P(h) with h = -2 g, P of degree 8 (relative error
//    2^-27.8); e ln 2 is added last.
//  * its square root by sqrtf.
//  * the angle 2 pi u1: its nearest quarter turn from the two top bits after
//    adding an eighth, the rest t in [-1/8, 1/8) exact; polynomials for
//    sin 2 pi t (2 pi in two parts) and cos 2 pi t, then swap and signs.
// Over all 2^23 u0, each with another u1, and all 2^23 u1, against FP64:
// relative error of a normal 4.5e-8 rms, 2.0e-7 at most, absolute error 4.4e-8
// rms; the same formula through logf, sqrtf and sincospif: 4.6e-8, 2.1e-7,
// 4.4e-8.  12.45e6 calls with Philox and their stores take 61.5 us, through
// CUDA's three functions 84.0.
PSGLD_HDI float4 normals4(uint4 x)
{
    // -2 ln u0
    const float m0 = as_float((x.x >> 9) | 0x3f800000u) - 0.99999994039535522f;
    const float m1 = as_float((x.z >> 9) | 0x3f800000u) - 0.99999994039535522f;
    const uint32_t e0 = (as_bits(m0) - 0x3f3504f3u) & 0xff800000u;   // sqrt(1/2)
    const uint32_t e1 = (as_bits(m1) - 0x3f3504f3u) & 0xff800000u;
    const float2 h = fma2(make_float2(as_float(as_bits(m0) - e0), as_float(as_bits(m1) - e1)), both(-2.0f), both(2.0f));
    // P's coefficients: those of (-2 ln(1 + g) / g + 2) / g in g, times (-1/2)^k / 4
    float2 q = both(0.1523810476064682f / 1024.0f);
    q = fma2(q, h, both(0.2582588195800781f / 512.0f));
    q = fma2(q, h, both(0.2649613618850708f / 256.0f));
    q = fma2(q, h, both(0.2836170792579651f / 128.0f));
    q = fma2(q, h, both(0.33216822147369385f / 64.0f));
    q = fma2(q, h, both(0.4000400900840759f / 32.0f));
    q = fma2(q, h, both(0.5000321865081787f / 16.0f));
    q = fma2(q, h, both(0.6666665077209473f / 8.0f));
    q = fma2(q, h, both(0.9999997615814209f / 4.0f));
    const float2 a = fma2(make_float2((float)(int32_t)e0, (float)(int32_t)e1), both(-1.6525916589735634e-07f),   // -2 ln 2 / 2^23
                          fma2(mul2(h, h), q, h));
    const float2 r = make_float2(sqrtf(a.x), sqrtf(a.y));
    // sin and cos of 2 pi u1
    const uint32_t w0 = x.y + 0x20000000u, w1 = x.w + 0x20000000u;
    const float2 t = fma2(make_float2(as_float(((w0 >> 7) & 0x007ffffcu) | 0x3f800000u),
                                      as_float(((w1 >> 7) & 0x007ffffcu) | 0x3f800000u)),
                          both(0.25f), both(-0.37499994039535522f));   // 2^-24 - 1/4 - 1/8
    const float2 z = mul2(t, t);
    float2 p = fma2(both(-75.36840057373047f), z, both(81.59188079833984f));
    p = fma2(p, z, both(-41.34165954589844f));
    p = fma2(p, z, both(-1.9520483363066887e-07f));
    const float2 sn = fma2(t, both(6.2831854820251465f), mul2(t, p));
    float2 c = fma2(both(58.62105941772461f), z, both(-85.42452239990234f));
    c = fma2(c, z, both(64.93914794921875f));
    c = fma2(c, z, both(-19.739208221435547f));
    c = fma2(c, z, both(1.0f));
    const bool o0 = w0 & 0x40000000u, o1 = w1 & 0x40000000u;   // an odd quarter: swap
    const float2 rc = mul2(r, make_float2(o0 ? sn.x : c.x, o1 ? sn.y : c.y));
    const float2 rs = mul2(r, make_float2(o0 ? c.x : sn.x, o1 ? c.y : sn.y));
    auto sign = [](float v, uint32_t w) { return as_float(as_bits(v) ^ (w & 0x80000000u)); };
    return make_float4(sign(rc.x, w0 + 0x40000000u), sign(rs.x, w0), sign(rc.y, w1 + 0x40000000u), sign(rs.y, w1));
}

}  // namespace dev
}  // namespace psgld
