// psgld_units.cu -- one PSGLD iteration on sparse data with few entries per
// row, as a gradient and an update launch per factor.
//
// The form for contexts whose rows hold few entries of a part, and for small
// ones of large K (step_by_units): most of the work is the Langevin step of
// rows with hardly an entry, which wants a flat pass over the factors at full
// occupancy rather than rows held by teams of lanes (psgld_rows.cu).
//
// Kernel 1, gradient.  A side's entries of the part, in row order, are cut
// into units of E consecutive entries, one warp per unit at a time: the other
// factor's rows are gathered into shared memory by bulk copies, mu and the
// Tweedie factor are formed one lane per entry, and the gradient is summed by
// row segments of the unit.  A row whose entries span several units publishes
// the sums of its pieces to per-unit head and tail slots, which the update
// adds in unit order, so the result does not depend on scheduling.
//
// Kernel 2, update.  A flat, coalesced pass over every (row, float4 group)
// item: the row's gradient (nothing for an empty row), noise, prior, step,
// mirror; reads X_cur, writes X_next.
//
// Sweeps of 3 10^5 x 5000, 1.2 10^6 entries, B = 16, at K = 16, 48, 100: 365,
// 873, 1841 us, with CUDA's logf, sqrtf and sincospif in the normals 395, 963,
// 1905; one launch of psgld_rows.cu: 532, 1064, 2314.
#include <algorithm>
#include <cstring>
#include <vector>

#include "psgld_slots.cuh"
#include "psgld_update.cuh"

namespace psgld {
namespace {

using dev::add4;
using dev::ldg4;
using dev::zero4;

constexpr int kThreads = 256;        // update kernel
constexpr int kGradThreads = 128;    // gradient kernel: four warps, one unit each

struct GradSide {
    const float *X_cur;    // own rows (n_rows x ldk)
    const float *Y_cur;    // gathered rows of the other factor
    float *Gout;           // this side's rows of G
    const int32_t *own;    // own row of each entry
    const int32_t *idx;    // other index of each entry
    const float *val;
    float *partial;        // 2 x units x ldk: head / tail partial sums
    int64_t base;          // first entry of the part
    int64_t n;             // entries of the part
    int64_t units;         // ceil(n / E)
    const uint16_t *Y16;   // BF16 copy of Y_cur (rows of ld16), gathered instead of it
    int prefetch_own;      // 1: own rows go to L2 with the gathers (own factor beyond L2)
};

struct GradParams {
    GradSide side[2];
    int ldk, lds, ngroups;    // row length, shared-memory row stride (floats), float4 groups
    int ld16, lds16;          // BF16 gathers: row length and shared-memory row stride (elements)
    float phi_inv, p, mu_min;
    int p_mode;               // 0: p = 0, 1: p = 1, 2: p = 2, 3: other
    int *err;                 // set to 16 when a bulk copy wait runs out
    uint32_t wait_polls;      // > 0: the first wait's poll limit (no suspension), for tests
};

struct UpdSide {
    const float *X_cur;
    float *X_next;
    const float *Gin;
    const int32_t *ptr;       // this part's row offsets (absolute entry indices)
    const float *partial;     // head / tail partial sums of the gradient kernel
    int64_t base;             // first entry of the part
    int64_t items;            // n_rows * ngroups (0 when the factor is frozen)
    uint16_t *X16_next;       // BF16 copy of X_next (rows of ld16)
    float prior_a, prior_b;   // d log p(x)/dx = prior_a + prior_b * x
};

struct UpdParams {
    UpdSide side[2];
    StepNoise noise;
    int K, ldk, ld16, ngroups, unit_shift;
    uint32_t div_magic;       // ceil(2^32 / ngroups) when item * ngroups < 2^32, else 0
};

__device__ __forceinline__ float dot4(const float4 a, const float4 b, float acc)
{
    acc = fmaf(a.x, b.x, acc);
    acc = fmaf(a.y, b.y, acc);
    acc = fmaf(a.z, b.z, acc);
    acc = fmaf(a.w, b.w, acc);
    return acc;
}

__device__ __forceinline__ void axpy4(float4 &acc, float e, const float4 y)
{
    acc.x = fmaf(e, y.x, acc.x);
    acc.y = fmaf(e, y.y, acc.y);
    acc.z = fmaf(e, y.z, acc.z);
    acc.w = fmaf(e, y.w, acc.w);
}

// Tweedie factor: e = (v - mu) * max(mu, mu_min)^(-p) / phi
__device__ __forceinline__ float tweedie_e(const GradParams &P, float v, float mu)
{
    const float d = v - mu;
    if (P.p_mode == 0) return d * P.phi_inv;
    const float mc = fmaxf(mu, P.mu_min);
    if (P.p_mode == 1) return d / mc * P.phi_inv;
    if (P.p_mode == 2) return d / (mc * mc) * P.phi_inv;
    return d * exp2f(-P.p * log2f(mc)) * P.phi_inv;
}

constexpr uint32_t kWaitLimit = 1u << 24;          // mbarrier polls before giving up
constexpr long long kWaitCycles = 1ll << 31;         // ... or about one second of SM clock
constexpr uint32_t kWaitHintNs = 2000;               // suspension per poll

__device__ __forceinline__ uint32_t smem_addr(const void *p)
{
    return (uint32_t)__cvta_generic_to_shared(p);
}

__device__ __forceinline__ void mbar_init(uint64_t *bar)
{
    asm volatile("mbarrier.init.shared::cta.b64 [%0], 1;" :: "r"(smem_addr(bar)) : "memory");
    asm volatile("fence.mbarrier_init.release.cluster;" ::: "memory");
}

__device__ __forceinline__ void mbar_expect_tx(uint64_t *bar, uint32_t bytes)
{
    asm volatile("mbarrier.arrive.expect_tx.shared::cta.b64 _, [%0], %1;"
                 :: "r"(smem_addr(bar)), "r"(bytes) : "memory");
}

// Waits (suspended, up to about `hint_ns`) for phase `parity` of the barrier
// to complete; true once it has.  The suspension keeps waiting warps from
// taking issue slots while the copies are in flight.
__device__ __forceinline__ bool mbar_try_wait(uint64_t *bar, uint32_t parity, uint32_t hint_ns)
{
    uint32_t ok;
    asm volatile("{\n\t.reg .pred p;\n\t"
                 "mbarrier.try_wait.parity.shared::cta.b64 p, [%1], %2, %3;\n\t"
                 "selp.u32 %0, 1, 0, p;\n\t}"
                 : "=r"(ok) : "r"(smem_addr(bar)), "r"(parity), "r"(hint_ns) : "memory");
    return ok != 0;
}

// One poll of phase `parity` of the barrier, without suspending.
__device__ __forceinline__ bool mbar_test_wait(uint64_t *bar, uint32_t parity)
{
    uint32_t ok;
    asm volatile("{\n\t.reg .pred p;\n\t"
                 "mbarrier.test_wait.parity.shared::cta.b64 p, [%1], %2;\n\t"
                 "selp.u32 %0, 1, 0, p;\n\t}"
                 : "=r"(ok) : "r"(smem_addr(bar)), "r"(parity) : "memory");
    return ok != 0;
}

// Bulk copy of `bytes` (a multiple of 16, both addresses 16-byte aligned)
// from global to this CTA's shared memory, completing on `bar`.
__device__ __forceinline__ void bulk_g2s(void *dst, const void *src, uint32_t bytes, uint64_t *bar)
{
    asm volatile("cp.async.bulk.shared::cluster.global.mbarrier::complete_tx::bytes [%0], [%1], %2, [%3];"
                 :: "r"(smem_addr(dst)), "l"(src), "r"(bytes), "r"(smem_addr(bar)) : "memory");
}

// Bulk prefetch of `bytes` (a multiple of 16, 16-byte aligned) into L2.
__device__ __forceinline__ void prefetch_l2(const void *src, uint32_t bytes)
{
    asm volatile("cp.async.bulk.prefetch.L2.global [%0], %1;" :: "l"(src), "r"(bytes) : "memory");
}

// q-th float4 group of row `row` of the warp's gathered rows: FP32 rows of
// `stride` floats, or (BF) BF16 rows of `stride` elements.
template <bool BF>
__device__ __forceinline__ float4 ys4(const float *ys, int row, int q, int stride)
{
    if constexpr (BF) {
        const uint2 v = *reinterpret_cast<const uint2 *>(reinterpret_cast<const uint16_t *>(ys) + (size_t)row * stride + 4 * q);
        return make_float4(__uint_as_float(v.x << 16), __uint_as_float(v.x & 0xFFFF0000u),
                           __uint_as_float(v.y << 16), __uint_as_float(v.y & 0xFFFF0000u));
    } else {
        return *reinterpret_cast<const float4 *>(ys + (size_t)row * stride + 4 * q);
    }
}

// A unit's entries as each lane loads them, one unit ahead of its work:
// lane l entry l (own row, other index, value); `edge` is, on lane 0, the
// own row of the entry just before the unit and, on lane 1, of the entry
// just after it (-1: none).
struct UnitIn {
    int own, jj;
    float vv;
    int edge;
};

template <int SID, int E>
__device__ __forceinline__ UnitIn load_unit(const GradParams &P, int64_t u)
{
    const GradSide &Sd = P.side[SID];
    const int lane32 = threadIdx.x & 31;
    const int64_t e0 = Sd.base + u * E, rem = Sd.n - u * E;
    UnitIn r{-1, 0, 0.f, -1};
    if (lane32 < E && lane32 < rem) {
        r.own = __ldg(Sd.own + e0 + lane32);
        r.jj = __ldg(Sd.idx + e0 + lane32);
        r.vv = __ldg(Sd.val + e0 + lane32);
    }
    if (lane32 == 0 && u > 0) r.edge = __ldg(Sd.own + e0 - 1);
    if (lane32 == 1 && rem > E) r.edge = __ldg(Sd.own + e0 + E);
    return r;
}

// One unit (E consecutive entries of side SID's part order) on one warp; SID
// is a template parameter so that the side's fields are fixed parameter
// offsets.  BF: the gathered rows are the BF16 copies (half the bytes;
// products and sums stay FP32).  `bar` completes once per unit, phase
// `parity`.  False when the gathers did not land in time (the warp stops).
template <int SID, int S, int NG, int E, bool BF>
__device__ __forceinline__ bool grad_unit(const GradParams &P, int64_t u, const UnitIn &in, float *ys,
                                          float *es, int *ow, int *sg, uint64_t *bar, uint32_t parity)
{
    constexpr int R = 32 / S;      // sub-teams per warp
    constexpr int NGP = S * NG;    // float4 groups a sub-team covers (>= ngroups)
    const int lane32 = threadIdx.x & 31;
    const int ng = P.ngroups, ldk = P.ldk, lds = BF ? P.lds16 : P.lds;
    const GradSide &Sd = P.side[SID];
    const int n = (int)(Sd.n - u * E < E ? Sd.n - u * E : E);

    // ---- 1. this lane's entry (loaded with the previous unit)
    const bool valid = lane32 < n;
    const int own = in.own, jj = in.jj;
    const float vv = in.vv;
    const int prev_own = __shfl_sync(0xffffffffu, in.edge, 0);   // rows of the entries just outside the unit
    const int next_own = __shfl_sync(0xffffffffu, in.edge, 1);
    const uint32_t row_bytes = BF ? (uint32_t)P.ld16 * 2u : (uint32_t)ldk * 4u;

    // ---- 2. bulk gathers into shared memory, once every lane is done with
    // the previous unit's (its reads ordered before the copies' writes)
    asm volatile("fence.proxy.async.shared::cta;" ::: "memory");
    __syncwarp();
    if (lane32 == 0) mbar_expect_tx(bar, (uint32_t)n * row_bytes);
    __syncwarp();
    bool done = false;
    if (P.wait_polls) {
        // a test limit: at most wait_polls polls, without suspending, made
        // before the copies are issued -- so the wait surely runs out
        for (uint32_t it = 0; it < P.wait_polls && !done; ++it) done = mbar_test_wait(bar, parity);
    }
    if (valid) {
        if constexpr (BF)
            bulk_g2s(reinterpret_cast<uint16_t *>(ys) + (size_t)lane32 * lds, Sd.Y16 + (int64_t)jj * P.ld16, row_bytes, bar);
        else
            bulk_g2s(ys + (size_t)lane32 * lds, Sd.Y_cur + (int64_t)jj * ldk, row_bytes, bar);
    }
    // each row segment's own row on its way to L2 while the gathers land
    const int own_prev_lane = __shfl_up_sync(0xffffffffu, own, 1);
    const bool seg_start = valid && (lane32 == 0 || own != own_prev_lane);
    if (seg_start && Sd.prefetch_own) prefetch_l2(Sd.X_cur + (int64_t)own * ldk, (uint32_t)ldk * 4u);
    // the first XP float4 groups of this lane's own row, loaded before the
    // wait (the rest after it, in the mu loop)
    constexpr int XP = NGP < 8 ? NGP : 8;
    float4 xp[XP];
    const float *xrow = Sd.X_cur + (int64_t)(valid ? own : 0) * ldk;
#pragma unroll
    for (int w = 0; w < XP; ++w) xp[w] = (valid && w < ng) ? ldg4(xrow + 4 * w) : zero4();
    const long long t_start = clock64();
    if (!P.wait_polls) {
        for (uint32_t it = 0; it < kWaitLimit && !done && clock64() - t_start < kWaitCycles; ++it)
            done = mbar_try_wait(bar, parity, kWaitHintNs);
    }
    if (!__all_sync(0xffffffffu, done)) {
        // The copies did not land: report it, wait (bounded again) for them
        // so that no copy targets freed shared memory, and give up.
        if (lane32 == 0) atomicOr(P.err, 16);
        const long long t_again = clock64();
        for (uint32_t it = 0; it < kWaitLimit && !done && clock64() - t_again < kWaitCycles; ++it)
            done = mbar_try_wait(bar, parity, kWaitHintNs);
        return false;
    }

    // ---- 3. mu and the Tweedie factor, one lane per entry
    float e = 0.f;
    if (valid) {
        const float *x = Sd.X_cur + (int64_t)own * ldk;
        float d = 0.f;
#pragma unroll
        for (int q = 0; q < NGP; ++q)
            if (q < ng) d = dot4(q < XP ? xp[q < XP ? q : 0] : ldg4(x + 4 * q), ys4<BF>(ys, lane32, q, lds), d);
        e = tweedie_e(P, vv, d);
    }
    const unsigned smask = __ballot_sync(0xffffffffu, seg_start);
    if (lane32 < E) {
        es[lane32] = e;
        ow[lane32] = own;
    }
    // sg[k]: the unit's entry that starts row segment k; sg[nseg] = n
    if (seg_start) sg[__popc(smask & ((1u << lane32) - 1u))] = lane32;
    if (lane32 == 0) sg[__popc(smask)] = n;
    __syncwarp();

    // ---- 4./5. gradient sums per row segment
    const int sub = lane32 / S, lane = lane32 & (S - 1);
    const int nseg = __popc(smask);
    float4 acc[NG];
    if (nseg == 1) {
        // one row: sub-team s takes entries s, s+R, ...; then add the sub-teams
#pragma unroll
        for (int g = 0; g < NG; ++g) acc[g] = zero4();
#pragma unroll 4
        for (int sl = sub; sl < n; sl += R) {
            const float es_ = es[sl];
#pragma unroll
            for (int g = 0; g < NG; ++g) {
                const int q = lane + g * S;
                if (q < ng) axpy4(acc[g], es_, ys4<BF>(ys, sl, q, lds));
            }
        }
#pragma unroll
        for (int o = S; o < 32; o <<= 1)
#pragma unroll
            for (int g = 0; g < NG; ++g) {
                acc[g].x += __shfl_xor_sync(0xffffffffu, acc[g].x, o);
                acc[g].y += __shfl_xor_sync(0xffffffffu, acc[g].y, o);
                acc[g].z += __shfl_xor_sync(0xffffffffu, acc[g].z, o);
                acc[g].w += __shfl_xor_sync(0xffffffffu, acc[g].w, o);
            }
        const int row = ow[0];
        float *dst = prev_own == row ? Sd.partial + head_slot(u, ldk)
                   : next_own == row ? Sd.partial + tail_slot(u, ldk)
                                     : Sd.Gout + (int64_t)row * ldk;
        if (sub == 0) {
#pragma unroll
            for (int g = 0; g < NG; ++g) {
                const int q = lane + g * S;
                if (q < ng) *reinterpret_cast<float4 *>(dst + 4 * q) = acc[g];
            }
        }
    } else {
        // several rows: sub-team s takes segments s, s+R, ...
        for (int k = sub; k < nseg; k += R) {
            const int st = sg[k], en = sg[k + 1];
            const int row = ow[st];
#pragma unroll
            for (int g = 0; g < NG; ++g) acc[g] = zero4();
#pragma unroll 4
            for (int sl = st; sl < en; ++sl) {
                const float es_ = es[sl];
#pragma unroll
                for (int g = 0; g < NG; ++g) {
                    const int q = lane + g * S;
                    if (q < ng) axpy4(acc[g], es_, ys4<BF>(ys, sl, q, lds));
                }
            }
            float *dst = (k == 0 && prev_own == row) ? Sd.partial + head_slot(u, ldk)
                       : (k == nseg - 1 && next_own == row) ? Sd.partial + tail_slot(u, ldk)
                                                             : Sd.Gout + (int64_t)row * ldk;
#pragma unroll
            for (int g = 0; g < NG; ++g) {
                const int q = lane + g * S;
                if (q < ng) *reinterpret_cast<float4 *>(dst + 4 * q) = acc[g];
            }
        }
    }
    return true;
}

// Each warp takes units u, u + T, u + 2T, ... (T = warps of the grid: a
// grid of one CTA per 4 units gives every warp one unit; a smaller grid
// keeps warps resident over several), loading the next unit's entries
// before working on the current one.
template <int S, int NG, int E, bool BF>
__global__ void __launch_bounds__(kGradThreads) grad_kernel(const __grid_constant__ GradParams P)
{
    extern __shared__ float4 smem4[];
    const int warp = threadIdx.x >> 5;
    const int lds = P.lds;
    constexpr int kWarpsPerCta = kGradThreads / 32;
    float *base = reinterpret_cast<float *>(smem4);
    float *ys = base + (size_t)warp * E * lds;                      // E gathered rows
    float *es = base + (size_t)kWarpsPerCta * E * lds + warp * E;   // e of each entry
    int *ow = reinterpret_cast<int *>(base + (size_t)kWarpsPerCta * E * lds + kWarpsPerCta * E) + warp * E;
    int *sg = reinterpret_cast<int *>(base + (size_t)kWarpsPerCta * (E * lds + 2 * E)) + warp * (E + 1);
    uint64_t *bar = reinterpret_cast<uint64_t *>(base + (size_t)kWarpsPerCta * (E * lds + 3 * E + 1)) + warp;

    const int64_t U0 = P.side[0].units, U = U0 + P.side[1].units;
    const int64_t T = (int64_t)gridDim.x * kWarpsPerCta;
    int64_t u = (int64_t)blockIdx.x * kWarpsPerCta + warp;
    if (u >= U) return;   // warp-uniform
    if ((threadIdx.x & 31) == 0) mbar_init(bar);
    __syncwarp();
    UnitIn cur = u < U0 ? load_unit<0, E>(P, u) : load_unit<1, E>(P, u - U0);
    for (uint32_t parity = 0; u < U; u += T, parity ^= 1u) {
        const int64_t nu = u + T;
        UnitIn nxt{-1, 0, 0.f, -1};
        if (nu < U) nxt = nu < U0 ? load_unit<0, E>(P, nu) : load_unit<1, E>(P, nu - U0);
        const bool ok = u < U0 ? grad_unit<0, S, NG, E, BF>(P, u, cur, ys, es, ow, sg, bar, parity)
                               : grad_unit<1, S, NG, E, BF>(P, u - U0, cur, ys, es, ow, sg, bar, parity);
        if (!ok) return;
        cur = nxt;
    }
}

// One (row, float4 group) item of factor SID (0 = W, 1 = H^T): items and
// factor offsets in 32 bits (step_by_units checks the sizes), slots in 64.
template <int SID, bool BF>
__device__ __forceinline__ void update_item32(const UpdParams &P, uint32_t item, float eps, float sd,
                                              uint32_t t_lo, uint32_t t_hi)
{
    const UpdSide &Sd = P.side[SID];
    const uint32_t ng = (uint32_t)P.ngroups;
    const uint32_t row = P.div_magic ? __umulhi(item, P.div_magic) : item / ng;
    const uint32_t q = item - row * ng;
    const uint32_t off = row * (uint32_t)P.ldk + 4u * q;
    const float4 x = ldg4(Sd.X_cur + off);
    float4 g = zero4();
    const int p0 = __ldg(Sd.ptr + row) - (int)Sd.base, p1 = __ldg(Sd.ptr + row + 1) - (int)Sd.base;
    if (p1 > p0) {
        const int u0 = p0 >> P.unit_shift, u1 = (p1 - 1) >> P.unit_shift;
        if (u0 == u1) {
            g = ldg4(Sd.Gin + off);
        } else {
            // the row's first unit's tail slot, then the later units' head slots, in unit order
            g = __ldcg(reinterpret_cast<const float4 *>(Sd.partial + tail_slot(u0, P.ldk) + 4u * q));
            const float *hp = Sd.partial + 4u * q;
            int uu = u0 + 1;
            for (; uu + 8 <= u1 + 1; uu += 8) {   // eight independent loads in flight
                float4 v[8];
#pragma unroll
                for (int w = 0; w < 8; ++w)
                    v[w] = __ldcg(reinterpret_cast<const float4 *>(hp + head_slot(uu + w, P.ldk)));
#pragma unroll
                for (int w = 0; w < 8; ++w) add4(g, v[w]);
            }
            for (; uu <= u1; ++uu) add4(g, __ldcg(reinterpret_cast<const float4 *>(hp + head_slot(uu, P.ldk))));
        }
    }
    const float4 z = dev::normals4(dev::philox(make_uint4(q, row, t_lo, (t_hi << 1) | (uint32_t)SID), P.noise.rk0,
                                               P.noise.rk1));
    float4 o = dev::langevin4(P.noise, Sd.prior_a, Sd.prior_b, x, g, z, eps, sd);
    dev::mask_padding(o, q, (uint32_t)P.K);
    *reinterpret_cast<float4 *>(Sd.X_next + off) = o;
    if constexpr (BF) {
        const __nv_bfloat162 a = __floats2bfloat162_rn(o.x, o.y), b = __floats2bfloat162_rn(o.z, o.w);
        *reinterpret_cast<uint2 *>(Sd.X16_next + (int64_t)row * P.ld16 + 4u * q) =
            make_uint2(*reinterpret_cast<const uint32_t *>(&a), *reinterpret_cast<const uint32_t *>(&b));
    }
}

template <bool BF>
__global__ void __launch_bounds__(kThreads, 5) units_update_kernel(const __grid_constant__ UpdParams P)
{
    const StepNoise &N = P.noise;
    const int64_t t = N.t_dev ? *N.t_dev + N.t_add : N.t_add;
    float eps = N.eps, sd = N.sd;
    if (N.eps_tab) {
        const float2 e = __ldg(N.eps_tab + (N.t_add - 1));
        eps = e.x;
        sd = e.y;
    }
    const uint32_t t_lo = (uint32_t)(uint64_t)t, t_hi = (uint32_t)((uint64_t)t >> 32);
    const uint32_t n0 = (uint32_t)P.side[0].items, n1 = (uint32_t)P.side[1].items;
    const uint32_t stride = gridDim.x * kThreads;
    uint32_t a = blockIdx.x * kThreads + threadIdx.x;
    for (; a < n0; a += stride) update_item32<0, BF>(P, a, eps, sd, t_lo, t_hi);
    for (a -= n0; a < n1; a += stride) update_item32<1, BF>(P, a, eps, sd, t_lo, t_hi);
}

using GradFn = void (*)(GradParams);

struct Shape {
    int S, NG, E, lds;
};

// Sub-team lanes S and float4 groups per lane NG cover K; E entries per unit
// keep a warp's shared memory (E gathered rows) near 17 KB at most; the row
// stride is padded so that its float4 count is odd (each lane reading its own
// row hits distinct banks).
Shape shape_for(int ngroups)
{
    Shape sh;
    if (ngroups <= 4) {            // K <= 16: one float4 group per lane
        sh.S = 1;
        while (sh.S < ngroups) sh.S <<= 1;
        sh.NG = 1;
    } else {                       // two groups per lane, up to 32 lanes
        sh.S = 4;
        while (sh.S * 2 < ngroups && sh.S < 32) sh.S <<= 1;
        sh.NG = (ngroups + sh.S - 1) / sh.S;
    }
    sh.E = ngroups <= 32 ? 32 : ngroups <= 64 ? 16 : 8;
    sh.lds = (ngroups & 1) ? 4 * ngroups : 4 * ngroups + 4;
    return sh;
}

template <bool BF>
GradFn pick_grad_t(const Shape &sh)
{
    if (sh.NG == 1) {
        switch (sh.S) {
        case 1: return grad_kernel<1, 1, 32, BF>;
        case 2: return grad_kernel<2, 1, 32, BF>;
        case 4: return grad_kernel<4, 1, 32, BF>;
        }
    }
    if (sh.NG == 2) {
        switch (sh.S) {
        case 4: return grad_kernel<4, 2, 32, BF>;
        case 8: return grad_kernel<8, 2, 32, BF>;
        case 16: return grad_kernel<16, 2, 32, BF>;
        case 32: return grad_kernel<32, 2, 16, BF>;
        }
    }
    if (sh.S == 32) {
        switch (sh.NG) {
        case 3: return grad_kernel<32, 3, 8, BF>;
        case 4: return grad_kernel<32, 4, 8, BF>;
        }
    }
    return nullptr;
}

// bf: the variant that gathers the BF16 copies of the factors
GradFn pick_grad(const Shape &sh, bool bf) { return bf ? pick_grad_t<true>(sh) : pick_grad_t<false>(sh); }

// Shared-memory stride of the BF16 rows: lds16 / 8 odd, so that the lanes'
// 8-byte reads of distinct rows spread over the banks.
int lds16_for(int ldk)
{
    const int m = gather_ld16(ldk) / 8;
    return 8 * ((m & 1) ? m : m + 1);
}

size_t grad_smem(const Shape &sh)
{
    const int warps = kGradThreads / 32;
    return sizeof(float) * (size_t)warps * ((size_t)sh.E * sh.lds + 3 * sh.E + 1) +
           sizeof(uint64_t) * warps;
}

}  // namespace

int unit_entries(int ngroups) { return shape_for(ngroups).E; }

// Two regions, on FP32 gathers, from sweeps of 12 shapes at K = 16 to 500
// (us, units / rows; `rho`: a row's entries of a part on average):
//   large factors and few entries per row, where most of the work is the
//   flat update, the more so the more of a row's lanes are padding.  2.1 10^5
//   rows, rho 1.5, K = 16, 20, 64, 96: 750 / 799, 860 / 1189, 1769 / 1958,
//   2933 / 2667; 2.5 10^5 rows, rho 3.2, K = 20, 32, 72, 96: 2112 / 2575,
//   2535 / 2629, 5405 / 5595, 6470 / 5679; 8 10^4 rows, rho 3.9, K = 36:
//   811 / 886, K = 64: 1119 / 965; 5.5 10^4 rows, rho 14.5, K = 72:
//   1242 / 1157.  Up to K = 8 a row is one or two lanes: rows as fast, but for
//   the largest factors: 3.05 10^5 rows, rho 0.5, K = 4: 192 / 232; 4.98 10^5
//   rows, rho 0.5, K = 8: 1358 / 1703.  Smaller factors where padding counts:
//   8 10^4 rows, rho 1.0, K = 20: 382 / 446, K = 36: rho 0.5 605 / 581, rho 4
//   828 / 910; 3.5 10^4 rows, K = 36, rho 4: 117 / 134.  From K = 65 to 256
//   padding counts for less: 1.5 10^5 rows, rho 2, K = 100, 200: 1421 / 1195,
//   2605 / 2027.
//   K > 96 and few entries in a part, where a launch is as long as one
//   warp's walk over a row with a hundred entries.  1600 rows, 25 000 entries,
//   K = 128, 200: 49 / 66, 81 / 115; 35 000 rows, 31 000 entries, 429 / 455,
//   584 / 763; 28 000 rows, 62 000 entries, 487 / 457, 715 / 784;
//   K = 300: 25 000 entries 137 / 123, 2500 59 / 117.
// With BF16 gathers the rows' gathers cost half as much and the flat update
// pays on the largest factors alone: 3.05 10^5 rows, rho 0.4, K = 16, 20, 50,
// 96: 373 / 518, 448 / 906, 1039 / 1624, 1697 / 2088; rho 1.5 525 / 430,
// 683 / 784, 1490 / 1271, 2328 / 1755; 4.98 10^5 rows, rho 1.0, K = 16, 72:
// 2614 / 4169, 10007 / 11659; and where 5 or 6 of a row's 8 lanes work:
// 8 10^4 rows, rho 0.8, K = 20: 408 / 455; 10^5 rows, rho 0.4: 119 / 143.
// Items and factor offsets in 32 bits.
bool step_by_units(int64_t I, int64_t J, int ngroups, int64_t nnz, int B, bool bf16)
{
    const int64_t rows = I + J, items = rows * ngroups, lim = (1ll << 31) - 1;
    if (items > lim || std::max(I, J) * 4 * ngroups > lim) return false;
    const double padding = (double)rows_groups(ngroups) / ngroups - 1.0;
    const double rho = 2.0 * (double)nnz / ((double)B * (double)rows);
    if (rows > 1 << 18 && ngroups < 32 && rho < (ngroups <= 16 ? 2.4e-6 : 1.8e-6) * (double)rows + padding) return true;
    if ((ngroups == 5 || ngroups == 6) && rows > 1 << 16 && rho < 2.0) return true;
    if (bf16) return false;
    if (ngroups == 9 && rows > 1 << 15 && rho >= 2.0 && rho < 6.0) return true;
    if (ngroups > 24 && nnz < (ngroups <= 64 ? 1536ll : 128ll) * ngroups * B) return true;
    if (ngroups <= 2 || items <= (1 << 19)) return false;
    return rho < (ngroups <= 16 ? 2.0 : 1.0) + (ngroups <= 16 || ngroups > 64 ? 4.0 : 2.0) * padding;
}

// CTAs of kernel `f` (`threads` threads, `smem` bytes of dynamic shared
// memory each) resident at once on the current device: SMs x CTAs per SM,
// remembered per host thread for the last two kernels asked about (the
// gradient kernels of one context, FP32 and BF16 gathers).
static int64_t resident_wave(const void *f, int threads, size_t smem)
{
    struct Entry {
        const void *f;
        int threads;
        size_t smem;
        int dev;
        int64_t wave;
    };
    thread_local Entry memo[2] = {{nullptr, 0, 0, -1, 0}, {nullptr, 0, 0, -1, 0}};
    thread_local int next = 0;
    int dev = 0;
    if (cudaGetDevice(&dev) != cudaSuccess) return 1ll << 40;
    for (const Entry &e : memo)
        if (e.f == f && e.threads == threads && e.smem == smem && e.dev == dev) return e.wave;
    int sms = 0, per_sm = 0;
    if (cudaDeviceGetAttribute(&sms, cudaDevAttrMultiProcessorCount, dev) != cudaSuccess ||
        cudaOccupancyMaxActiveBlocksPerMultiprocessor(&per_sm, f, threads, smem) != cudaSuccess ||
        sms <= 0 || per_sm <= 0)
        return 1ll << 40;   // unknown: no cap
    memo[next] = {f, threads, smem, dev, (int64_t)sms * per_sm};
    next ^= 1;
    return (int64_t)sms * per_sm;
}

psgld_status prepare_units(psgld_ctx *c)
{
    const Shape sh = shape_for(c->ngroups);
    for (int bf = 0; bf < 2; ++bf) {
        const GradFn fn = pick_grad(sh, bf != 0);
        if (!fn) return fail(c, PSGLD_ERR_ARG, "unsupported K");
        PSGLD_CK(c, cudaFuncSetAttribute(fn, cudaFuncAttributeMaxDynamicSharedMemorySize, (int)grad_smem(sh)));
    }
    return side_stream(c);
}

psgld_status launch_units(psgld_ctx *c, int part, int64_t t, const int64_t *t_dev, int64_t t_add, cudaStream_t st,
                          cudaEvent_t mid, unsigned rec_flags)
{
    const Shape sh = shape_for(c->ngroups);
    const bool bf = gather_bf16(c);
    const GradFn fn = pick_grad(sh, bf);
    const bool upd[2] = {!c->opt.freeze_W, !c->opt.freeze_H};
    GradParams GP{};
    UpdParams UP{};
    for (int s = 0; s < 2; ++s) {
        const SideLayout &L = c->side[s];
        GradSide &Gs = GP.side[s];
        UpdSide &Us = UP.side[s];
        const int64_t n_rows = s == 0 ? c->I : c->J;
        const int64_t base = L.part_first[part], n = L.part_first[part + 1] - base;
        Gs.X_cur = s == 0 ? c->W[c->wcur] : c->Ht[c->hcur];
        Gs.Y_cur = s == 0 ? c->Ht[c->hcur] : c->W[c->wcur];
        Gs.Gout = c->G + (s == 0 ? 0 : c->I * c->ldk);
        Gs.own = L.own;
        Gs.idx = L.idx;
        Gs.val = L.val;
        Gs.partial = L.unit_sums;
        Gs.base = base;
        Gs.n = n;
        Gs.units = upd[s] ? (n + sh.E - 1) / sh.E : 0;
        if (bf) {
            Gs.Y16 = s == 0 ? c->H16[c->hcur] : c->W16[c->wcur];
            Us.X16_next = s == 0 ? c->W16[c->wcur ^ 1] : c->H16[c->hcur ^ 1];
        }
        Gs.prefetch_own = 4.0 * (double)n_rows * c->ldk > 64.0 * (1 << 20);
        Us.X_cur = Gs.X_cur;
        Us.X_next = s == 0 ? c->W[c->wcur ^ 1] : c->Ht[c->hcur ^ 1];
        Us.Gin = Gs.Gout;
        Us.ptr = L.ptr + (int64_t)part * n_rows;
        Us.partial = L.unit_sums;
        Us.base = base;
        Us.items = upd[s] ? n_rows * c->ngroups : 0;
        if (c->prior.kind == PSGLD_PRIOR_EXPONENTIAL) {
            Us.prior_a = (float)-(s == 0 ? c->prior.lambda_w : c->prior.lambda_h);
        } else {
            const double sg = s == 0 ? c->prior.sigma_w : c->prior.sigma_h;
            Us.prior_b = (float)(-1.0 / (sg * sg));
        }
    }
    GP.ldk = c->ldk;
    GP.lds = sh.lds;
    GP.ld16 = gather_ld16(c->ldk);
    GP.lds16 = lds16_for(c->ldk);
    GP.ngroups = c->ngroups;
    GP.phi_inv = (float)(1.0 / c->phi);
    GP.p = (float)c->p;
    GP.mu_min = (float)c->opt.mu_min;
    GP.p_mode = c->p == 0.0 ? 0 : c->p == 1.0 ? 1 : c->p == 2.0 ? 2 : 3;
    GP.err = c->kflag;
    GP.wait_polls = (uint32_t)c->opt.debug_wait_polls;
    fill_noise(c, part, t, t_dev, t_add, UP.noise);
    UP.K = c->K;
    UP.ldk = c->ldk;
    UP.ld16 = GP.ld16;
    UP.ngroups = c->ngroups;
    UP.unit_shift = sh.E == 32 ? 5 : sh.E == 16 ? 4 : 3;
    const int64_t max_items = std::max(UP.side[0].items, UP.side[1].items);
    UP.div_magic = (max_items * c->ngroups < (1ll << 32))
                       ? (uint32_t)(((1ull << 32) + c->ngroups - 1) / c->ngroups) : 0u;
    auto update = [&](int side, cudaStream_t ss) {     // side 2: both
        UpdParams U = UP;
        if (side < 2) U.side[side ^ 1].items = 0;
        const int64_t n = U.side[0].items + U.side[1].items;
        const int grid = (int)std::min<int64_t>((n + kThreads - 1) / kThreads, 152 * 16);
        if (grid > 0) (bf ? units_update_kernel<true> : units_update_kernel<false>)<<<grid, kThreads, 0, ss>>>(U);
    };
    // resident: one wave of CTAs whose warps walk several units each (the
    // next unit's entries load during the current one); otherwise one unit
    // per warp, so that two launches on two streams share the SMs
    auto gradient = [&](int side, cudaStream_t ss, bool resident) {
        GradParams G = GP;
        if (side < 2) G.side[side ^ 1].units = 0;
        const int64_t n = G.side[0].units + G.side[1].units;
        int64_t grid = (n + kGradThreads / 32 - 1) / (kGradThreads / 32);
        if (resident) grid = std::min<int64_t>(grid, resident_wave((const void *)fn, kGradThreads, grad_smem(sh)));
        if (grid > 0) fn<<<(int)grid, kGradThreads, grad_smem(sh), ss>>>(G);
    };
    // W and H^T on two streams: within L2 (64 MB) each side's gradient, then
    // its update, so that the arithmetic of one side overlaps the gathers of
    // the other; beyond it the W side's gradient alone on the full grid, then
    // the H side's beside the W side's update.  Their outputs are disjoint, so
    // the result is the same bit for bit as in order on one stream, which
    // profiling and frozen factors take.  Inside a capture the fork and join
    // become graph edges.
    if (mid || !upd[0] || !upd[1]) {
        gradient(2, st, true);
        if (mid) PSGLD_CK(c, cudaEventRecordWithFlags(mid, st, rec_flags));
        update(2, st);
        PSGLD_CK(c, cudaGetLastError());
        return PSGLD_OK;
    }
    const bool l2_fit = 4.0 * (double)(c->I + c->J) * c->ldk <= 64.0 * (1 << 20);
    if (!l2_fit) gradient(0, st, true);
    const psgld_status fs = fork_side(c, st);
    if (fs != PSGLD_OK) return fs;
    gradient(1, c->side_stream, !l2_fit);
    update(1, c->side_stream);
    if (l2_fit) gradient(0, st, false);
    update(0, st);
    PSGLD_CK(c, cudaGetLastError());
    return join_side(c, st);
}

}  // namespace psgld
