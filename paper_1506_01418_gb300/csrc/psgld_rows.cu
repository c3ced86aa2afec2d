// psgld_rows.cu -- one PSGLD iteration on sparse data in one launch.
//
// For part Pi_t every block (r, c) updates the W rows of row piece r and the
// H columns of column piece c from (W^(t-1), H^(t-1))  (Eq. psgld_w and
// Eq. psgld_h).  Because the B blocks of a part cover every row piece and
// every column piece exactly once, one iteration updates every row of W and
// every row of H^T:
//
//   w_i <- w_i + eps (S sum_{j in row i of Pi_t} e_ij h_j + dlog p(w_i)) + sqrt(2 eps) z
//   h_j <- h_j + eps (S sum_{i in col j of Pi_t} e_ij w_i + dlog p(h_j)) + sqrt(2 eps) z
//   e_ij = (v_ij - mu_ij) max(mu_ij, mu_min)^(-p) / phi,  mu_ij = w_i . h_j
//
// followed by |.| for non-negative models (Sec. 3.2).  This is the Tweedie
// gradient of Sec. 4 (d/dmu of -d_beta(v||mu)/phi with beta = 2 - p).
//
// A row of either factor needs only the old factors and its own entries of
// the part, and the new factors go to the other buffer of the ping-pong
// pair, so a row's gradient and its update are one piece of work with no
// wait between them: SDDMM, Tweedie factor, SpMM and Langevin step in
// registers, no gradient array in memory.
//
// A team of T lanes holds a factor row as NG float4 groups per lane (lane l
// the groups l, l + T, ...: a load of 16 T consecutive bytes).  Per entry the
// team loads the other factor's row, forms mu by a butterfly over its lanes,
// the Tweedie factor, and adds e y to the row's gradient; U entries go
// together, so that their loads are in flight at once and one butterfly and
// one Tweedie factor serve all of them.  Rows are shared out by their entries
// in the part:
//   light  (at most light_row): one team per row, 32 / T rows per warp;
//   mid    (at most kMidRow): one warp per row, its teams taking every
//          (32 / T)-th entry; the teams' sums are added by a butterfly and
//          each team updates its share of the row's groups;
//   heavy: a block per chunk of kChunk entries, its warps' sums added in
//          shared memory; of a row with several chunks the block that arrives
//          last adds the chunks' sums in order and updates the row.
// Light rows are found by walking all rows; the others are in two lists made
// with the layout.  The sums' order is fixed by the row's entries alone, so
// the result does not depend on scheduling.  Heavy rows go first, and the
// light and mid blocks alternate in the grid: the light rows of a large W
// are mostly the update's arithmetic and streaming, the mid rows mostly
// gathers, so each fills the issue slots that the other leaves.
//
// What bounds it: instructions and the latency of the gathers.  Of 10^8
// entries, K = 100, B = 64 (W beyond L2) a part-step's light rows without any
// entry take 119 us, 100 M warp instructions at 0.70 per cycle and scheduler,
// most of them Philox and the normals (their rows come into L2 a warp's share
// at a time, 3 % less than without).  Against the gradient and the update as
// two launches per side on two streams (before): 272 instead of 314 us a
// part-step there; 41.7 instead of 45.8 us with 10^7 entries, K = 50, B = 32
// (factors in L2); and one launch instead of four where launches count: a sweep
// of 256 x 256 dense counts, K = 8, B = 4, and its read-back 32 instead of 48 us.
// The factors are read by ordinary loads (launch_early); through the read-only
// path the two took 281 and 41.9 us with a cheaper square root in the normals.
// Thresholds measured on the first two then, ms a sweep with light up to 16,
// mid up to 128 and chunks of 512 18.0 and 1.34: 8, 128, 512: 18.3 and 1.43;
// 32, 128, 512: 18.4 and 1.44; 16, 96, 384: 18.9 and 1.37; 16, 192, 768: 18.2
// and 1.38.
#include <algorithm>
#include <cstring>
#include <vector>

#include "psgld_update.cuh"

namespace psgld {
namespace {

constexpr int kThreads = 256;
constexpr int kWarps = kThreads / 32;

struct RowSide {
    const float *X;            // own rows (n_rows x ldk)
    const float *Y;            // the other factor's rows
    float *Xn;                 // own rows after the step
    const uint16_t *Y16;       // BF16 copy of Y (rows of ld16), gathered instead of it
    uint16_t *Xn16;            // BF16 copy of Xn
    const int32_t *ptr;        // this part's row offsets (absolute entry indices)
    const int32_t *idx;        // other index of each entry
    const float *val;
    const int4 *mid;           // this part's mid rows (row, first entry, entries, 0)
    const int4 *heavy;         // ... and its heavy rows' chunks (row, first entry, entries, number)
    float *partial;            // a row of ldk sums per chunk
    int *arrived;              // per chunk: of a row's first one, the chunks done
    int n_rows, n_mid, n_heavy;   // zero when the factor is frozen
    int far;                   // 1: the own factor is beyond L2
    float prior_a, prior_b;       // d log p(x)/dx = prior_a + prior_b * x
};

struct RowParams {
    RowSide side[2];
    StepNoise noise;
    int K, ldk, ld16, ng;         // ng = ldk / 4 float4 groups
    int light;                    // most entries of a light row
    int iters;                    // light rows: row batches per warp
    int mid_blocks[2], light_blocks[2];
    uint32_t mid_share;           // floor(2^32 mid blocks / mid and light blocks)
    float phi_inv, p, mu_min;
    int p_mode;                   // 0: p = 0, 1: p = 1, 2: p = 2, 3: other
    int *err;
    uint32_t wait_polls;          // > 0: poll limit of the bounded-wait check (for tests)
};

// Tweedie factor: e = (v - mu) * max(mu, mu_min)^(-p) / phi
__device__ __forceinline__ float tweedie_e(const RowParams &P, float v, float mu)
{
    const float d = v - mu;
    if (P.p_mode == 0) return d * P.phi_inv;
    const float mc = fmaxf(mu, P.mu_min);
    if (P.p_mode == 1) return d / mc * P.phi_inv;
    if (P.p_mode == 2) return d / (mc * mc) * P.phi_inv;
    return d * exp2f(-P.p * log2f(mc)) * P.phi_inv;
}

__device__ __forceinline__ float2 lo2(const float4 a) { return make_float2(a.x, a.y); }
__device__ __forceinline__ float2 hi2(const float4 a) { return make_float2(a.z, a.w); }

// acc += a (elementwise) b, in pairs
__device__ __forceinline__ float4 fma4(float2 a_lo, float2 a_hi, const float4 b, const float4 acc)
{
    const float2 l = dev::fma2(a_lo, lo2(b), lo2(acc)), h = dev::fma2(a_hi, hi2(b), hi2(acc));
    return make_float4(l.x, l.y, h.x, h.y);
}

__device__ __forceinline__ float4 shfl_xor4(const float4 a, int o)
{
    return make_float4(__shfl_xor_sync(0xffffffffu, a.x, o), __shfl_xor_sync(0xffffffffu, a.y, o),
                       __shfl_xor_sync(0xffffffffu, a.z, o), __shfl_xor_sync(0xffffffffu, a.w, o));
}

// Bulk prefetch of `bytes` (a multiple of 16, 16-byte aligned) into L2.
__device__ __forceinline__ void prefetch_l2(const void *src, uint32_t bytes)
{
    asm volatile("cp.async.bulk.prefetch.L2.global [%0], %1;" :: "l"(src), "r"(bytes) : "memory");
}

// A row read once, past L1 (which keeps the gathered rows).
__device__ __forceinline__ float4 ld_stream(const float *p)
{
    float4 v;
    asm volatile("ld.global.L1::no_allocate.v4.f32 {%0, %1, %2, %3}, [%4];"
                 : "=f"(v.x), "=f"(v.y), "=f"(v.z), "=f"(v.w) : "l"(p) : "memory");
    return v;
}

// From L2: sums that other blocks of this launch wrote.
__device__ __forceinline__ float4 ld_l2(const float *p)
{
    float4 v;
    asm volatile("ld.global.cg.v4.f32 {%0, %1, %2, %3}, [%4];"
                 : "=f"(v.x), "=f"(v.y), "=f"(v.z), "=f"(v.w) : "l"(p) : "memory");
    return v;
}

// What a team's lane holds of its row: all groups but the last are the
// row's in every lane; in the last, lanes past the row hold zeros (and read
// another group of the gathered rows).
template <int T, int NG>
struct Row {
    float4 x[NG], acc[NG];

    __device__ __forceinline__ void clear_acc()
    {
#pragma unroll
        for (int g = 0; g < NG; ++g) acc[g] = dev::zero4();
    }

    // src: this lane's first group; in_last: it has one in the last
    __device__ __forceinline__ void load(const float *src, bool in_last)
    {
#pragma unroll
        for (int g = 0; g < NG; ++g) x[g] = g + 1 < NG || in_last ? ld_stream(src + 4 * g * T) : dev::zero4();
        clear_acc();
    }
};

// U values, one per entry, summed over the team's lanes: halving butterflies
// that leave lane l with the sum of value l mod U, then whole ones.
template <int T, int U>
__device__ __forceinline__ float team_sum(float (&d)[U], int l)
{
    int n = U;
#pragma unroll
    for (int o = 1; o < U; o <<= 1) {
        n >>= 1;
#pragma unroll
        for (int k = 0; k < n; ++k) {
            const bool up = l & o;
            const float keep = up ? d[2 * k + 1] : d[2 * k], give = up ? d[2 * k] : d[2 * k + 1];
            d[k] = keep + __shfl_xor_sync(0xffffffffu, give, o);
        }
    }
#pragma unroll
    for (int o = U; o < T; o <<= 1) d[0] += __shfl_xor_sync(0xffffffffu, d[0], o);
    return d[0];
}

// The gathered rows as a lane reads them: its first group (lanes past a
// one-group row: the row's first), and its last.
template <int T, int NG, bool BF>
struct Source {
    const char *base, *last;
    uint32_t pitch;

    __device__ __forceinline__ Source(const RowParams &P, const RowSide &S, int l, bool in_last)
    {
        constexpr int kGroup = BF ? 8 : 16;
        pitch = (uint32_t)(BF ? P.ld16 * 2 : P.ldk * 4);
        base = BF ? reinterpret_cast<const char *>(S.Y16) : reinterpret_cast<const char *>(S.Y);
        base += NG > 1 || in_last ? l * kGroup : 0;
        last = in_last ? base + (NG - 1) * T * kGroup : base;
    }

    __device__ __forceinline__ void load(uint32_t j, float4 (&y)[NG]) const
    {
        constexpr int kGroup = BF ? 8 : 16;
        const char *row = base + (uint64_t)j * pitch;
#pragma unroll
        for (int g = 0; g < NG; ++g) {
            const char *at = g + 1 < NG || NG == 1 ? row + g * T * kGroup : last + (uint64_t)j * pitch;
            if constexpr (BF) {
                const uint2 w = *reinterpret_cast<const uint2 *>(at);
                y[g] = make_float4(__uint_as_float(w.x << 16), __uint_as_float(w.x & 0xFFFF0000u),
                                   __uint_as_float(w.y << 16), __uint_as_float(w.y & 0xFFFF0000u));
            } else {
                y[g] = *reinterpret_cast<const float4 *>(at);
            }
        }
    }
};

// T entries at a time, U of them together: entry c + l of the team has index
// j and value v in lane l; n: the team's entries; most: the most of the
// warp's teams, so that the butterflies run with full warps (entries past
// n weigh nothing).  fetch(c, j, v) brings entries c + l.
template <int T, int NG, int U, bool BF, class Fetch>
__device__ __forceinline__ void gather(const RowParams &P, const Source<T, NG, BF> &Y, Row<T, NG> &r, uint32_t n,
                                       uint32_t most, int l, int j, float v, Fetch fetch)
{
    for (uint32_t c = 0; c < most; c += T) {
        int jn = 0;
        float vn = 0.f;
        if (c + T < most) fetch(c + T, jn, vn);
        const uint32_t upto = most - c < T ? most - c : T;
#pragma unroll 1
        for (uint32_t t = 0; t < upto; t += U) {
            float4 y[U][NG];
#pragma unroll
            for (int u = 0; u < U; ++u) Y.load((uint32_t)__shfl_sync(0xffffffffu, j, t + u, T), y[u]);
            float d[U];
#pragma unroll
            for (int u = 0; u < U; ++u) {
                float2 s = dev::mul2(lo2(r.x[0]), lo2(y[u][0]));
                s = dev::fma2(hi2(r.x[0]), hi2(y[u][0]), s);
#pragma unroll
                for (int g = 1; g < NG; ++g) {
                    s = dev::fma2(lo2(r.x[g]), lo2(y[u][g]), s);
                    s = dev::fma2(hi2(r.x[g]), hi2(y[u][g]), s);
                }
                d[u] = s.x + s.y;
            }
            const uint32_t mine = t + (l & (U - 1));
            const float mu = team_sum<T, U>(d, l);
            const float vu = __shfl_sync(0xffffffffu, v, mine, T);
            const float w = c + mine < n ? tweedie_e(P, vu, mu) : 0.f;
#pragma unroll
            for (int u = 0; u < U; ++u) {
                const float2 e = dev::both(__shfl_sync(0xffffffffu, w, u, T));
#pragma unroll
                for (int g = 0; g < NG; ++g) r.acc[g] = fma4(e, e, y[u][g], r.acc[g]);
            }
        }
        j = jn;
        v = vn;
    }
}

// The warp's teams' sums added up, in every lane.
template <int T, int NG>
__device__ __forceinline__ void add_teams(Row<T, NG> &r)
{
#pragma unroll
    for (int o = T; o < 32; o <<= 1)
#pragma unroll
        for (int g = 0; g < NG; ++g) dev::add4(r.acc[g], shfl_xor4(r.acc[g], o));
}

struct Clock {
    float eps, sd;
    uint32_t t_lo, t_hi;
};

__device__ __forceinline__ Clock read_clock(const StepNoise &N)
{
    Clock c;
    const int64_t t = N.t_dev ? *N.t_dev + N.t_add : N.t_add;
    c.eps = N.eps;
    c.sd = N.sd;
    if (N.eps_tab) {
        const float2 e = N.eps_tab[N.t_add - 1];
        c.eps = e.x;
        c.sd = e.y;
    }
    c.t_lo = (uint32_t)(uint64_t)t;
    c.t_hi = (uint32_t)((uint64_t)t >> 32);
    return c;
}

// Group q of a row after the step, to `out` (and its BF16 copy).
template <bool BF>
__device__ __forceinline__ void store_group(const RowParams &P, const RowSide &S, int sid, const Clock &c,
                                            uint32_t row, int q, float4 x, float4 g, float *out)
{
    const float4 z = dev::normals4(dev::philox(make_uint4((uint32_t)q, row, c.t_lo, (c.t_hi << 1) | (uint32_t)sid),
                                               P.noise.rk0, P.noise.rk1));
    float4 o = dev::langevin4(P.noise, S.prior_a, S.prior_b, x, g, z, c.eps, c.sd);
    dev::mask_padding(o, (uint32_t)q, (uint32_t)P.K);
    *reinterpret_cast<float4 *>(out) = o;
    if constexpr (BF) {
        const __nv_bfloat162 a = __floats2bfloat162_rn(o.x, o.y), b = __floats2bfloat162_rn(o.z, o.w);
        *reinterpret_cast<uint2 *>(S.Xn16 + (int64_t)row * P.ld16 + 4 * q) =
            make_uint2(*reinterpret_cast<const uint32_t *>(&a), *reinterpret_cast<const uint32_t *>(&b));
    }
}

// ---- a bounded wait, for the test of the timeout path -----------------------
//
// The part-step waits for nothing but its own loads.  With wait_polls > 0
// each block first brings a row of the other factor into shared memory by a
// bulk copy on an mbarrier, polling (at most wait_polls times) before it
// issues the copy, so that the wait surely runs out: the error flag is set,
// the copy in flight is waited for with the normal limit, and the block
// returns without updating its rows.

constexpr uint32_t kWaitLimit = 1u << 24;     // mbarrier polls before giving up
constexpr long long kWaitCycles = 1ll << 31;  // ... or about one second of SM clock
constexpr uint32_t kWaitHintNs = 2000;        // suspension per poll

__device__ __forceinline__ uint32_t smem_addr(const void *p) { return (uint32_t)__cvta_generic_to_shared(p); }

__device__ bool gather_wait_check(const RowParams &P, const RowSide &S)
{
    __shared__ __align__(16) float row0[kMaxK];
    __shared__ uint64_t bar;
    __shared__ int landed;
    if (threadIdx.x == 0) {
        asm volatile("mbarrier.init.shared::cta.b64 [%0], 1;" :: "r"(smem_addr(&bar)) : "memory");
        asm volatile("fence.mbarrier_init.release.cluster;" ::: "memory");
        const uint32_t bytes = (uint32_t)P.ldk * 4u;
        asm volatile("mbarrier.arrive.expect_tx.shared::cta.b64 _, [%0], %1;"
                     :: "r"(smem_addr(&bar)), "r"(bytes) : "memory");
        uint32_t done = 0;
        for (uint32_t n = 0; n < P.wait_polls && !done; ++n)
            asm volatile("{\n\t.reg .pred p;\n\t"
                         "mbarrier.test_wait.parity.shared::cta.b64 p, [%1], 0;\n\t"
                         "selp.u32 %0, 1, 0, p;\n\t}" : "=r"(done) : "r"(smem_addr(&bar)) : "memory");
        asm volatile("cp.async.bulk.shared::cluster.global.mbarrier::complete_tx::bytes [%0], [%1], %2, [%3];"
                     :: "r"(smem_addr(row0)), "l"(S.Y), "r"(bytes), "r"(smem_addr(&bar)) : "memory");
        landed = (int)done;
        if (!done) atomicOr(P.err, 16);
        const long long t0 = clock64();
        for (uint32_t n = 0; n < kWaitLimit && !done && clock64() - t0 < kWaitCycles; ++n)
            asm volatile("{\n\t.reg .pred p;\n\t"
                         "mbarrier.try_wait.parity.shared::cta.b64 p, [%1], 0, %2;\n\t"
                         "selp.u32 %0, 1, 0, p;\n\t}" : "=r"(done) : "r"(smem_addr(&bar)), "r"(kWaitHintNs) : "memory");
    }
    __syncthreads();
    return landed != 0;
}

// U, UM: entries together in light rows, in the others.
template <int T, int NG, int U, int UM, bool BF, int MINB>
__global__ void __launch_bounds__(kThreads, MINB) rows_kernel(const __grid_constant__ RowParams P)
{
    constexpr int R = 32 / T;                       // teams per warp
    const int lane = threadIdx.x & 31, warp = threadIdx.x >> 5;
    const int l = lane & (T - 1), team = lane / T;
    const bool in_last = l + (NG - 1) * T < P.ng;
    const int n_heavy = P.side[0].n_heavy + P.side[1].n_heavy;
    dev::wait_prior();
    dev::let_next();
    if (P.wait_polls && !gather_wait_check(P, P.side[P.side[0].n_rows ? 0 : 1])) return;
    const Clock clk = read_clock(P.noise);
    Row<T, NG> r;
    int b = blockIdx.x;

    if (b < n_heavy) {                              // one chunk of a row, the whole block
        const int sid = b < P.side[0].n_heavy ? 0 : 1;
        const RowSide &S = P.side[sid];
        if (sid) b -= P.side[0].n_heavy;
        const int4 rec = __ldg(S.heavy + b);
        const uint32_t row = (uint32_t)rec.x, all = (uint32_t)rec.z;
        const int chunks = (int)((all + kChunk - 1) / kChunk);
        const uint32_t at0 = (uint32_t)rec.w * kChunk, c0 = (uint32_t)rec.y + at0;
        const uint32_t n = all - at0 < kChunk ? all - at0 : kChunk;
        r.load(S.X + (int64_t)row * P.ldk + 4 * l, in_last);
        constexpr uint32_t step = R * kWarps;       // entry i of team k of the block: i step + k
        const uint32_t k = warp * R + team;
        auto fetch = [&](uint32_t c, int &j, float &v) {
            const uint32_t i = (c + l) * step + k, at = c0 + (i < n ? i : n - 1);
            j = __ldg(S.idx + at);
            v = __ldg(S.val + at);
        };
        int j;
        float v;
        fetch(0, j, v);
        gather<T, NG, UM, BF>(P, Source<T, NG, BF>(P, S, l, in_last), r, (n + step - 1 - k) / step,
                              (n + step - 1) / step, l, j, v, fetch);
        add_teams(r);
        __shared__ float4 sums[kWarps][T * NG];
        __shared__ int last;
        if (team == 0) {
#pragma unroll
            for (int g = 0; g < NG; ++g) sums[warp][l + g * T] = r.acc[g];
        }
        __syncthreads();
        const int q = threadIdx.x;
        float4 s = dev::zero4();
        if (q < P.ng) {
            s = sums[0][q];
#pragma unroll
            for (int w = 1; w < kWarps; ++w) dev::add4(s, sums[w][q]);
        }
        if (chunks > 1) {
            // the row's sums go to its chunks' slots; the block that arrives
            // last adds them in chunk order
            if (q < P.ng) __stcg(reinterpret_cast<float4 *>(S.partial + (int64_t)b * P.ldk) + q, s);
            __threadfence();
            __syncthreads();
            const int first = b - rec.w;
            if (threadIdx.x == 0) {
                last = atomicAdd(S.arrived + first, 1) == chunks - 1;
                if (last) S.arrived[first] = 0;
            }
            __syncthreads();
            if (!last) return;
            __threadfence();
            if (q < P.ng) {
                s = dev::zero4();
                for (int i = 0; i < chunks; ++i)
                    dev::add4(s, ld_l2(S.partial + (int64_t)(first + i) * P.ldk + 4 * q));
            }
        }
        if (q < P.ng) {
            const int64_t off = (int64_t)row * P.ldk + 4 * q;
            store_group<BF>(P, S, sid, clk, row, q, dev::ld4(S.X + off), s, S.Xn + off);
        }
        return;
    }
    b -= n_heavy;
    const int m = (int)__umulhi((uint32_t)b, P.mid_share);   // mid blocks before this one
    if ((int)__umulhi((uint32_t)b + 1u, P.mid_share) > m) {  // one row per warp
        const int sid = m < P.mid_blocks[0] ? 0 : 1;
        const RowSide &S = P.side[sid];
        const int at = (sid ? m - P.mid_blocks[0] : m) * kWarps + warp;
        if (at >= S.n_mid) return;
        const int4 rec = __ldg(S.mid + at);
        const uint32_t row = (uint32_t)rec.x, p0 = (uint32_t)rec.y, n = (uint32_t)rec.z;
        const int64_t off = (int64_t)row * P.ldk + 4 * l;
        r.load(S.X + off, in_last);
        auto fetch = [&](uint32_t c, int &j, float &v) {   // entry i of team k: i R + k
            const uint32_t i = (c + l) * R + team, e = p0 + (i < n ? i : n - 1);
            j = __ldg(S.idx + e);
            v = __ldg(S.val + e);
        };
        int j;
        float v;
        fetch(0, j, v);
        gather<T, NG, UM, BF>(P, Source<T, NG, BF>(P, S, l, in_last), r, (n + R - 1 - team) / R, (n + R - 1) / R, l,
                              j, v, fetch);
        add_teams(r);
        // team k takes groups k, k + R, ... of each lane: every lane draws
        // noise, where one team would draw NG times
#pragma unroll
        for (int k = 0; k < NG; k += R) {
            float4 x = r.x[k], s = r.acc[k];
            int g = k;
#pragma unroll
            for (int i = 1; i < R && k + i < NG; ++i)
                if (team == i) {
                    x = r.x[k + i];
                    s = r.acc[k + i];
                    g = k + i;
                }
            if (team < (NG - k < R ? NG - k : R) && (g + 1 < NG || in_last))
                store_group<BF>(P, S, sid, clk, row, l + g * T, x, s, S.Xn + off + 4 * g * T);
        }
        return;
    }
    // one row per team, `iters` batches of R rows per warp; the next batch's
    // row offsets and first entries load during the current one
    const int lb = b - m;
    const int sid = lb < P.light_blocks[0] ? 0 : 1;
    const RowSide &S = P.side[sid];
    const uint32_t n_rows = (uint32_t)S.n_rows, light = (uint32_t)P.light;
    uint32_t row = (uint32_t)((sid ? lb - P.light_blocks[0] : lb) * kWarps + warp) * R * P.iters + team;
    const Source<T, NG, BF> Y(P, S, l, in_last);
    const int32_t *ptr = S.ptr + row;
    const float *src = S.X + (int64_t)row * P.ldk + 4 * l;
    float *dst = S.Xn + (int64_t)row * P.ldk + 4 * l;
    uint32_t p = 0, n = 0xffffffffu;                // no row: as one that is not light
    int j = 0;
    float v = 0.f;
    auto next_row = [&]() {
        n = 0xffffffffu;
        if (row < n_rows) {
            p = __ldg(ptr);
            n = __ldg(ptr + 1) - p;
        }
    };
    auto fetch = [&](uint32_t first, uint32_t count, uint32_t c, int &jj, float &vv) {
        const uint32_t i = c + l, e = first + (i < count ? i : count - 1);
        if (count) {
            jj = __ldg(S.idx + e);
            vv = __ldg(S.val + e);
        }
    };
    if (S.far && lane == 0 && row < n_rows) {
        const uint32_t left = n_rows - row, mine = (uint32_t)(R * P.iters);
        prefetch_l2(S.X + (int64_t)row * P.ldk, (left < mine ? left : mine) * (uint32_t)P.ldk * 4u);
    }
    next_row();
    if (n <= light) fetch(p, n, 0, j, v);
    for (int it = 0; it < P.iters; ++it) {
        const uint32_t row0 = row, p0 = p;
        const bool on = n <= light;
        const uint32_t n0 = on ? n : 0u;
        const int j0 = j;
        const float v0 = v;
        if (on) r.load(src, in_last);
        else r.clear_acc();
        row += R;
        ptr += R;
        if (it + 1 < P.iters) {
            next_row();
            if (n <= light) fetch(p, n, 0, j, v);
        }
        const uint32_t most = __reduce_max_sync(0xffffffffu, n0);
        if (most) {
            gather<T, NG, U, BF>(P, Y, r, n0, most, l, j0, v0,
                                 [&](uint32_t c, int &jj, float &vv) { fetch(p0, n0, c, jj, vv); });
            if (!n0) r.clear_acc();                 // nothing of the other teams' weightless entries
        }
        if (on) {
#pragma unroll
            for (int g = 0; g < NG; ++g)
                if (g + 1 < NG || in_last)
                    store_group<BF>(P, S, sid, clk, row0, l + g * T, r.x[g], r.acc[g], dst + 4 * g * T);
        }
        src += R * P.ldk;
        dst += R * P.ldk;
    }
}

using RowFn = void (*)(RowParams);

struct RowKernel {
    int T;
    int groups;     // T lanes' float4 groups: ng and padding
    RowFn fn;
};

template <int T, int NG, int U, int UM, bool BF, int MINB>
RowKernel rows() { return {T, T * NG, rows_kernel<T, NG, U, UM, BF, MINB>}; }

// Lanes per team and groups per lane for ng float4 groups, entries together
// (light rows, others), and blocks per SM to hold the registers to.  Warps in
// flight count most: 64 registers give 32 per SM, which two groups a lane and
// two entries together fit but for 40 to 64 bytes of spills.  Sweeps of 10^8 entries, K = 100 (and of 3 10^7,
// BF16): 16 x 2 with 2 entries 18.0 (13.6) ms, with 4 in 80 registers 18.6
// (14.3), 32 x 1 19.2 (14.2), 8 x 4 in 114 registers (16 warps) 24.7; of 10^7,
// K = 50: 8 x 2 with 2 entries 1.34 ms, 16 x 1 with 4 1.37, with 2 1.46.
// A third group in 80 registers pays where it saves padding: 7 10^4 x 10^4,
// 5 10^6 entries, B = 32 at K = 36: 4 x 3 886 us, 8 x 2 959; at K = 72, 96:
// 8 x 3 1270, 1309, 16 x 2 1493, 1560; at K = 20, 32: 8 x 1 with 4 entries
// 644, 654 us, with 2 704, 716.
template <bool BF>
RowKernel pick_rows(int ng)
{
    if (ng <= 1) return rows<1, 1, 1, 1, BF, 4>();
    if (ng <= 2) return rows<2, 1, 2, 2, BF, 4>();
    if (ng <= 4) return rows<4, 1, 2, 4, BF, 4>();
    if (ng <= 8) return rows<8, 1, 4, 4, BF, 4>();
    if (ng <= 12) return rows<4, 3, 2, 2, BF, 3>();
    if (ng <= 16) return rows<8, 2, 2, 2, BF, 4>();
    if (ng <= 24) return rows<8, 3, 2, 2, BF, 3>();
    if (ng <= 32) return rows<16, 2, 2, 2, BF, 4>();
    if (ng <= 48) return rows<16, 3, 1, 2, BF, 3>();
    if (ng <= 64) return rows<32, 2, 2, 2, BF, 4>();
    if (ng <= 96) return rows<32, 3, 1, 2, BF, 3>();
    return rows<32, 4, 1, 2, BF, 2>();
}

// BF16 copy of an n x ldk FP32 factor into rows of ld16 (padding zero)
__global__ void gather_copy_kernel(const float *__restrict__ X, int64_t n, int ldk, int ld16,
                                   uint16_t *__restrict__ Y)
{
    const int64_t total = n * ld16;
    for (int64_t a = blockIdx.x * (int64_t)blockDim.x + threadIdx.x; a < total;
         a += (int64_t)gridDim.x * blockDim.x) {
        const int64_t r = a / ld16;
        const int k = (int)(a - r * ld16);
        const float x = k < ldk ? X[r * ldk + k] : 0.f;
        const __nv_bfloat16 b = __float2bfloat16_rn(x);
        Y[a] = *reinterpret_cast<const uint16_t *>(&b);
    }
}

}  // namespace

int gather_ld16(int ldk) { return 8 * ((ldk + 7) / 8); }

int rows_groups(int ng) { return pick_rows<false>(ng).groups; }

bool gather_bf16(const psgld_ctx *c) { return c->opt.gather_bf16 && !c->dense && c->W16[0] && c->H16[1]; }

psgld_status build_gather_shadows(psgld_ctx *c, cudaStream_t st)
{
    if (!c->opt.gather_bf16 || c->dense || !c->has_factors) return PSGLD_OK;
    const int ld16 = gather_ld16(c->ldk);
    for (int side = 0; side < 2; ++side) {
        const int64_t n = side == 0 ? c->I : c->J;
        const float *X = side == 0 ? c->W[c->wcur] : c->Ht[c->hcur];
        for (int b = 0; b < 2; ++b) {   // both of the pair: the part-step writes all but the padding
            uint16_t *&Y = side == 0 ? c->W16[b] : c->H16[b];
            if (!Y) {
                Y = static_cast<uint16_t *>(dev_alloc(c, sizeof(uint16_t) * (size_t)std::max<int64_t>(n * ld16, 1), st));
                if (!Y) return fail(c, PSGLD_ERR_OOM, "device allocation failed");
            }
            const unsigned grid = (unsigned)std::max<int64_t>(1, std::min<int64_t>((n * ld16 + 255) / 256, 152 * 16));
            gather_copy_kernel<<<grid, 256, 0, st>>>(X, n, c->ldk, ld16, Y);
            PSGLD_CK(c, cudaGetLastError());
        }
    }
    return PSGLD_OK;
}

psgld_status launch_rows(psgld_ctx *c, int part, int64_t t, const int64_t *t_dev, int64_t t_add, cudaStream_t st)
{
    const bool bf = gather_bf16(c);
    const bool upd[2] = {!c->opt.freeze_W, !c->opt.freeze_H};
    const RowKernel k = bf ? pick_rows<true>(c->ngroups) : pick_rows<false>(c->ngroups);
    const int R = 32 / k.T;
    RowParams P{};
    for (int s = 0; s < 2; ++s) {
        const SideLayout &L = c->side[s];
        RowSide &S = P.side[s];
        const int64_t n_rows = s == 0 ? c->I : c->J;
        S.X = s == 0 ? c->W[c->wcur] : c->Ht[c->hcur];
        S.Y = s == 0 ? c->Ht[c->hcur] : c->W[c->wcur];
        S.Xn = s == 0 ? c->W[c->wcur ^ 1] : c->Ht[c->hcur ^ 1];
        if (bf) {
            S.Y16 = s == 0 ? c->H16[c->hcur] : c->W16[c->wcur];
            S.Xn16 = s == 0 ? c->W16[c->wcur ^ 1] : c->H16[c->hcur ^ 1];
        }
        S.far = 4.0 * (double)n_rows * c->ldk > 64.0 * (1 << 20);
        S.ptr = L.ptr + (int64_t)part * n_rows;
        S.idx = L.idx;
        S.val = L.val;
        S.mid = L.mid + L.mid_first[part];
        S.heavy = L.heavy + L.heavy_first[part];
        S.partial = L.partial;
        S.arrived = L.arrived;
        if (upd[s]) {
            S.n_rows = (int)n_rows;
            S.n_mid = (int)(L.mid_first[part + 1] - L.mid_first[part]);
            S.n_heavy = (int)(L.heavy_first[part + 1] - L.heavy_first[part]);
        }
        if (c->prior.kind == PSGLD_PRIOR_EXPONENTIAL) {
            S.prior_a = (float)-(s == 0 ? c->prior.lambda_w : c->prior.lambda_h);
        } else {
            const double sg = s == 0 ? c->prior.sigma_w : c->prior.sigma_h;
            S.prior_b = (float)(-1.0 / (sg * sg));
        }
    }
    P.light = c->light_row;
    const int64_t rows = (int64_t)P.side[0].n_rows + P.side[1].n_rows;
    // light rows: up to eight row batches per warp, fewer while the grid
    // would not give every SM eight blocks
    P.iters = (int)std::max<int64_t>(1, std::min<int64_t>(8, rows / ((int64_t)kWarps * R * 152 * 8)));
    const int64_t per_block = (int64_t)kWarps * R * P.iters;
    int64_t mid = 0, light = 0;
    for (int s = 0; s < 2; ++s) {
        P.mid_blocks[s] = (P.side[s].n_mid + kWarps - 1) / kWarps;
        P.light_blocks[s] = (int)((P.side[s].n_rows + per_block - 1) / per_block);
        mid += P.mid_blocks[s];
        light += P.light_blocks[s];
    }
    if (mid + light > 0) P.mid_share = (uint32_t)std::min<uint64_t>(((uint64_t)mid << 32) / (uint64_t)(mid + light) + 1, 0xffffffffu);
    const int64_t grid = (int64_t)P.side[0].n_heavy + P.side[1].n_heavy + mid + light;
    P.K = c->K;
    P.ldk = c->ldk;
    P.ld16 = gather_ld16(c->ldk);
    P.ng = c->ngroups;
    P.phi_inv = (float)(1.0 / c->phi);
    P.p = (float)c->p;
    P.mu_min = (float)c->opt.mu_min;
    P.p_mode = c->p == 0.0 ? 0 : c->p == 1.0 ? 1 : c->p == 2.0 ? 2 : 3;
    P.err = c->kflag;
    P.wait_polls = (uint32_t)c->opt.debug_wait_polls;
    fill_noise(c, part, t, t_dev, t_add, P.noise);
    if (grid > 0) PSGLD_CK(c, launch_early(!c->opt.profile, k.fn, (unsigned)grid, kThreads, 0, st, P));
    PSGLD_CK(c, cudaGetLastError());
    return PSGLD_OK;
}

}  // namespace psgld
