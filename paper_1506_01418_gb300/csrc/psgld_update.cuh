// psgld_update.cuh -- the Langevin update of one factor entry and its noise,
// shared by the sparse part-step (psgld_rows.cu) and the dense path's update
// kernels (psgld_step.cu):
//   x <- x + eps (S g + dlog p(x)) + sqrt(2 eps) z,  then |.| for
// non-negative models (Sec. 3 Eq. psgld_w, Eq. psgld_h; Sec. 3.2).
#pragma once

#include <cmath>

#include "psgld_internal.cuh"
#include "psgld_normals.cuh"

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
