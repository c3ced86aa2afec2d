// psgld_update.cuh -- the Langevin update of one factor entry and its noise,
// shared by the sparse part-step (psgld_rows.cu) and the dense path's update
// kernels (psgld_step.cu):
//   x <- x + eps (S g + dlog p(x)) + sqrt(2 eps) z,  then |.| for
// non-negative models (Sec. 3 Eq. psgld_w, Eq. psgld_h; Sec. 3.2).
#pragma once

#include <cmath>

#include "psgld_internal.cuh"

namespace psgld {

// What every row of one iteration shares.
struct StepNoise {
    const int64_t *t_dev;        // if non-null, t = *t_dev + t_add
    int64_t t_add;
    const float2 *eps_tab;       // captured sweeps with eps_t: (eps, sqrt(2 eps)) of each part-step
    float eps, sd, S;            // step, sqrt(2 eps), N / |Pi_t|
    int mirror;                  // 1: x <- |x|
    uint32_t rk0[10], rk1[10];   // Philox round keys (seed + r * Weyl constants)
};

// Noise and step parameters of iteration t (part `part`) of context c; with
// t_dev the kernels read t from *t_dev + t_add (captured graphs), and
// eps_t = (a / t)^b from the table that the sweep's first launch fills.
void fill_noise(const psgld_ctx *c, int part, int64_t t, const int64_t *t_dev, int64_t t_add, StepNoise &N);

namespace dev {

// An ordinary load: for factors and gradients in kernels that launch_early
// starts (see there).  ldg4 is for plain launches.
__device__ __forceinline__ float4 ld4(const float *p) { return *reinterpret_cast<const float4 *>(p); }

__device__ __forceinline__ float4 ldg4(const float *p) { return __ldg(reinterpret_cast<const float4 *>(p)); }

__device__ __forceinline__ float4 zero4() { return make_float4(0.f, 0.f, 0.f, 0.f); }

__device__ __forceinline__ void add4(float4 &a, const float4 b)
{
    a.x += b.x; a.y += b.y; a.z += b.z; a.w += b.w;
}

// Two FP32 operations per instruction (the sm_100 family's packed FP32
// arithmetic), each rounded like its scalar form.
__device__ __forceinline__ float2 fma2(float2 a, float2 b, float2 c)
{
    float2 d;
    asm("fma.rn.f32x2 %0, %1, %2, %3;"
        : "=l"(reinterpret_cast<unsigned long long &>(d))
        : "l"(reinterpret_cast<unsigned long long &>(a)), "l"(reinterpret_cast<unsigned long long &>(b)),
          "l"(reinterpret_cast<unsigned long long &>(c)));
    return d;
}

__device__ __forceinline__ float2 mul2(float2 a, float2 b)
{
    float2 d;
    asm("mul.rn.f32x2 %0, %1, %2;"
        : "=l"(reinterpret_cast<unsigned long long &>(d))
        : "l"(reinterpret_cast<unsigned long long &>(a)), "l"(reinterpret_cast<unsigned long long &>(b)));
    return d;
}

__device__ __forceinline__ float2 both(float x) { return make_float2(x, x); }

// Four normals from four random words: uniforms on (0, 1), u = the top 23
// bits plus one half, times 2^-23 (exact in FP32); Box-Muller on (u0, u1)
// and (u2, u3), cos first, then sin.
//
// Instructions bound every kernel that draws noise, so the two pairs go
// through packed arithmetic, and each function is written for the arguments
// it meets here (no subnormals, no infinities, no large angles):
//  * u0: the bits under the exponent of 1 give 1 + m 2^-23; subtracting
//    1 - 2^-24 is exact.
//  * -2 ln u0: u0 = 2^e (1 + g), g in [sqrt(1/2) - 1, sqrt(2) - 1];
//    -2 ln(1 + g) = h + h^2 P(h) with h = -2 g, P the minimax polynomial of
//    degree 8 (relative error 2^-27.8, by linear programming on Chebyshev
//    nodes); e ln 2 is added last.
//  * the square root: the hardware's reciprocal square root times its
//    argument, and one Newton step on the residual.
//  * the angle 2 pi u1: its nearest quarter turn from the two top bits after
//    adding an eighth, the rest t in [-1/8, 1/8) exact; minimax polynomials
//    for sin 2 pi t (2 pi in two parts) and cos 2 pi t, then swap and signs.
// Measured over all 2^23 u0, each with another u1, against FP64: relative
// error of a normal 4.5e-8 rms, 2.0e-7 at most, absolute error 4.4e-8 rms;
// the same formula through logf, sqrtf and sincospif: 4.6e-8, 2.1e-7, 4.4e-8.
// With Philox, 115 instructions per call against 195; 12.45e6 calls and
// their stores 57.6 against 82.3 us.
__device__ __forceinline__ float4 normals4(uint4 x)
{
    // -2 ln u0
    const float m0 = __uint_as_float((x.x >> 9) | 0x3f800000u) - 0.99999994039535522f;
    const float m1 = __uint_as_float((x.z >> 9) | 0x3f800000u) - 0.99999994039535522f;
    const uint32_t e0 = (__float_as_uint(m0) - 0x3f3504f3u) & 0xff800000u;
    const uint32_t e1 = (__float_as_uint(m1) - 0x3f3504f3u) & 0xff800000u;
    const float2 h = fma2(make_float2(__uint_as_float(__float_as_uint(m0) - e0), __uint_as_float(__float_as_uint(m1) - e1)),
                          both(-2.0f), both(2.0f));
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
    const float2 a = fma2(make_float2((float)(int)e0, (float)(int)e1), both(-1.6525916589735634e-07f),   // -2 ln 2 / 2^23
                          fma2(mul2(h, h), q, h));
    // its square root
    float y0, y1;
    asm("rsqrt.approx.f32 %0, %1;" : "=f"(y0) : "f"(a.x));
    asm("rsqrt.approx.f32 %0, %1;" : "=f"(y1) : "f"(a.y));
    const float2 y = make_float2(y0, y1), s0 = mul2(a, y);
    const float2 r = fma2(fma2(make_float2(-s0.x, -s0.y), s0, a), mul2(y, both(0.5f)), s0);
    // sin and cos of 2 pi u1
    const uint32_t w0 = x.y + 0x20000000u, w1 = x.w + 0x20000000u;
    const float2 t = fma2(make_float2(__uint_as_float(((w0 >> 7) & 0x007ffffcu) | 0x3f800000u),
                                      __uint_as_float(((w1 >> 7) & 0x007ffffcu) | 0x3f800000u)),
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
    auto sign = [](float v, uint32_t w) { return __uint_as_float(__float_as_uint(v) ^ (w & 0x80000000u)); };
    return make_float4(sign(rc.x, w0 + 0x40000000u), sign(rs.x, w0), sign(rc.y, w1 + 0x40000000u), sign(rs.y, w1));
}

// Philox4x32-10 (Salmon et al., SC'11) with the round keys precomputed on the
// host: each round multiplies words 0 and 2 into 64-bit products and mixes
// their high halves with words 1, 3 and the round key.
__device__ __forceinline__ uint4 philox(uint4 c, const uint32_t (&rk0)[10], const uint32_t (&rk1)[10])
{
#pragma unroll
    for (int r = 0; r < 10; ++r) {
        const uint64_t p0 = (uint64_t)0xD2511F53u * c.x;
        const uint64_t p1 = (uint64_t)0xCD9E8D57u * c.z;
        c = make_uint4((uint32_t)(p1 >> 32) ^ c.y ^ rk0[r], (uint32_t)p1,
                       (uint32_t)(p0 >> 32) ^ c.w ^ rk1[r], (uint32_t)p0);
    }
    return c;
}

// x + eps (S g + dlog p(x)) + sqrt(2 eps) z, d log p(x)/dx = prior_a +
// prior_b x, mirrored for non-negative models.
__device__ __forceinline__ float4 langevin4(const StepNoise &N, float prior_a, float prior_b, float4 x, float4 g,
                                            float4 z, float eps, float sd)
{
    auto two = [&](float2 xx, float2 gg, float2 zz) {
        return fma2(both(sd), zz,
                    fma2(both(eps), fma2(both(N.S), gg, fma2(both(prior_b), xx, both(prior_a))), xx));
    };
    const float2 lo = two(make_float2(x.x, x.y), make_float2(g.x, g.y), make_float2(z.x, z.y));
    const float2 hi = two(make_float2(x.z, x.w), make_float2(g.z, g.w), make_float2(z.z, z.w));
    if (N.mirror) return make_float4(fabsf(lo.x), fabsf(lo.y), fabsf(hi.x), fabsf(hi.y));
    return make_float4(lo.x, lo.y, hi.x, hi.y);
}

// The padding entries (k >= K) of group q stay zero.
__device__ __forceinline__ void mask_padding(float4 &o, uint32_t q, uint32_t K)
{
    const uint32_t k0 = 4u * q;
    if (k0 + 4u > K) {
        if (k0 + 1 >= K) o.y = 0.f;
        if (k0 + 2 >= K) o.z = 0.f;
        if (k0 + 3 >= K) o.w = 0.f;
    }
}

}  // namespace dev
}  // namespace psgld
