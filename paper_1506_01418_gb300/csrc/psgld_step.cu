// psgld_step.cu -- one PSGLD iteration (Algorithm 1's loop body), and the
// update kernels of the dense tensor-core path.
//
// On sparse data an iteration is one launch (psgld_rows.cu) or, with few
// entries per row, a gradient and an update launch per factor
// (psgld_units.cu).  On dense data kept for the tensor cores (dense_path) it is two: the likelihood gradient
// G of every row of W and H^T (psgld_dense.cu), then the update here, a
// flat, fully coalesced pass over every (row, float4 group) item of both
// factors: the row's gradient, Philox4x32-10 normals (counter = group, row,
// t, matrix), prior gradient, step, mirror; reads X_cur, writes X_next
// (ping-pong buffers, so no row is read and written by the same launch).
// Philox's integer multiplies and Box-Muller make this ALU-bound, so it runs
// at full lane occupancy rather than inside the tensor-core kernel.
#include <algorithm>
#include <cstring>
#include <vector>

#include "psgld_update.cuh"

namespace psgld {
namespace {

constexpr int kThreads = 256;        // update kernels

struct UpdSide {
    const float *X_cur;
    float *X_next;
    const float *Gin;
    int64_t items;            // n_rows * ngroups (0 when the factor is frozen)
    int64_t gstride;          // distance between partial gradient arrays
    int gparts;               // partial gradient arrays to add
    uint16_t *sh;             // two-sided dense kernel: BF16 shadow of X_next (else null)
    int64_t n_rows;           // I or J
    int sh_tiles;             // 64-row shadow tiles per piece
    float prior_a, prior_b;   // d log p(x)/dx = prior_a + prior_b * x
};

struct UpdParams {
    UpdSide side[2];
    StepNoise noise;
    int K, ldk, ngroups;
    uint32_t div_magic;       // ceil(2^32 / ngroups) when item * ngroups < 2^32, else 0
    int small;                // 1: every index below 2^31 (update_item_dense32)
    int eps_poly;             // 1: eps_t = (a/t)^b computed on the device (no table)
    double eps_a, eps_b;
    int B, sh_kp;             // pieces; shadow tile width (two-sided dense kernel)
};

// Step size and iteration of this launch.
__device__ __forceinline__ int64_t read_step(const UpdParams &P, float &eps, float &sd)
{
    const StepNoise &N = P.noise;
    const int64_t t = N.t_dev ? *N.t_dev + N.t_add : N.t_add;
    eps = N.eps;
    sd = N.sd;
    if (N.eps_tab) {
        const float2 e = N.eps_tab[N.t_add - 1];
        eps = e.x;
        sd = e.y;
    } else if (P.eps_poly) {
        const double e = pow(P.eps_a / (double)t, P.eps_b);
        eps = (float)e;
        sd = (float)sqrt(2.0 * e);
    }
    return t;
}

// One (row, float4 group) item of factor SID (0 = W, 1 = H^T); SID is a
// template parameter so that the side's fields are fixed parameter offsets.
template <int SID>
__device__ __forceinline__ void update_item(const UpdParams &P, int64_t item, float eps, float sd,
                                            uint32_t t_lo, uint32_t t_hi)
{
    const UpdSide &Sd = P.side[SID];
    const int ng = P.ngroups, ldk = P.ldk;
    const int64_t row = P.div_magic ? (int64_t)__umulhi((uint32_t)item, P.div_magic) : item / ng;
    const int q = (int)(item - row * ng);
    const int64_t off = row * ldk + 4 * q;
    const float4 x = dev::ld4(Sd.X_cur + off);
    // G, or the sum in M-tile order of the block's partial arrays
    float4 g = dev::ld4(Sd.Gin + off);
    for (int h = 1; h < Sd.gparts; ++h) dev::add4(g, dev::ld4(Sd.Gin + h * Sd.gstride + off));
    const float4 z = dev::box_muller4(dev::philox(make_uint4((uint32_t)q, (uint32_t)row, t_lo, (t_hi << 1) | (uint32_t)SID),
                                                  P.noise.rk0, P.noise.rk1));
    float4 o = dev::langevin4(P.noise, Sd.prior_a, Sd.prior_b, x, g, z, eps, sd);
    dev::mask_padding(o, (uint32_t)q, (uint32_t)P.K);
    *reinterpret_cast<float4 *>(Sd.X_next + off) = o;
    if (Sd.sh) dev::shadow_store4(Sd.sh, row, 4 * q, o, Sd.n_rows, P.B, Sd.sh_tiles, P.sh_kp);
}

__global__ void __launch_bounds__(kThreads, 5) update_kernel(const __grid_constant__ UpdParams P)
{
    dev::wait_prior();
    dev::let_next();
    float eps, sd;
    const int64_t t = read_step(P, eps, sd);
    const uint32_t t_lo = (uint32_t)(uint64_t)t, t_hi = (uint32_t)((uint64_t)t >> 32);
    // the flat item sequence: W items, then H^T items
    const int64_t n0 = P.side[0].items, n1 = P.side[1].items;
    const int64_t stride = (int64_t)gridDim.x * kThreads;
    int64_t a = blockIdx.x * (int64_t)kThreads + threadIdx.x;
    for (; a < n0; a += stride) update_item<0>(P, a, eps, sd, t_lo, t_hi);
    for (a -= n0; a < n1; a += stride) update_item<1>(P, a, eps, sd, t_lo, t_hi);
}

// The update of the dense path with 32-bit index arithmetic (items, factor
// and gradient offsets and the BF16 shadows' offsets all below 2^31,
// checked on the host): the same arithmetic, the same result bit for bit as
// update_item on the dense path, in fewer instructions.  The shadow's tile
// layout is dev::shadow_store4's, here in 32-bit offsets.
__device__ __forceinline__ void shadow_store4_32(uint16_t *sh, uint32_t row, uint32_t k0, float4 v, uint32_t n,
                                                 uint32_t B, uint32_t tiles, uint32_t KP)
{
    const uint32_t piece = ((row + 1u) * B - 1u) / n;
    const uint32_t rr = row - (piece * n) / B;
    const uint32_t rho = rr & 63u;
    const uint32_t kk = k0 & 63u, c = kk >> 3;
    const uint32_t off = (piece * tiles + (rr >> 6)) * 64u * KP + (k0 >> 6) * 4096u + rho * 64u +
                         ((c ^ (rho & 7u)) << 3) + (kk & 7u);
    __nv_bfloat162 lo = __floats2bfloat162_rn(v.x, v.y), hi = __floats2bfloat162_rn(v.z, v.w);
    *reinterpret_cast<uint2 *>(sh + off) =
        make_uint2(*reinterpret_cast<uint32_t *>(&lo), *reinterpret_cast<uint32_t *>(&hi));
}

template <int SID>
__device__ __forceinline__ void update_item_dense32(const UpdParams &P, uint32_t item, float eps, float sd,
                                                    uint32_t t_lo, uint32_t t_hi)
{
    const UpdSide &Sd = P.side[SID];
    const uint32_t ng = (uint32_t)P.ngroups;
    const uint32_t row = P.div_magic ? __umulhi(item, P.div_magic) : item / ng;
    const uint32_t q = item - row * ng;
    const uint32_t off = row * (uint32_t)P.ldk + 4u * q;
    const float4 x = dev::ld4(Sd.X_cur + off);
    // G, or the sum in M-tile order of the block's partial arrays
    float4 g = dev::ld4(Sd.Gin + off);
    for (int h = 1; h < Sd.gparts; ++h) dev::add4(g, dev::ld4(Sd.Gin + (uint32_t)h * (uint32_t)Sd.gstride + off));
    const float4 z = dev::box_muller4(dev::philox(make_uint4(q, row, t_lo, (t_hi << 1) | (uint32_t)SID),
                                                  P.noise.rk0, P.noise.rk1));
    float4 o = dev::langevin4(P.noise, Sd.prior_a, Sd.prior_b, x, g, z, eps, sd);
    dev::mask_padding(o, q, (uint32_t)P.K);
    *reinterpret_cast<float4 *>(Sd.X_next + off) = o;
    if (Sd.sh)
        shadow_store4_32(Sd.sh, row, 4u * q, o, (uint32_t)Sd.n_rows, (uint32_t)P.B, (uint32_t)Sd.sh_tiles,
                         (uint32_t)P.sh_kp);
}

__global__ void __launch_bounds__(kThreads, 5) update_kernel_dense32(const __grid_constant__ UpdParams P)
{
    dev::wait_prior();
    dev::let_next();
    float eps, sd;
    const int64_t t = read_step(P, eps, sd);
    const uint32_t t_lo = (uint32_t)(uint64_t)t, t_hi = (uint32_t)((uint64_t)t >> 32);
    const uint32_t n0 = (uint32_t)P.side[0].items, n1 = (uint32_t)P.side[1].items;
    const uint32_t stride = gridDim.x * kThreads;
    uint32_t a = blockIdx.x * kThreads + threadIdx.x;
    for (; a < n0; a += stride) update_item_dense32<0>(P, a, eps, sd, t_lo, t_hi);
    for (a -= n0; a < n1; a += stride) update_item_dense32<1>(P, a, eps, sd, t_lo, t_hi);
}

}  // namespace

void fill_noise(const psgld_ctx *c, int part, int64_t t, const int64_t *t_dev, int64_t t_add, StepNoise &N)
{
    N.t_dev = t_dev;
    N.t_add = t_dev ? t_add : t;
    const bool poly = c->opt.eps_mode == PSGLD_EPS_POLY;
    N.eps_tab = poly && t_dev ? c->eps_tab : nullptr;
    const double eps = poly && !t_dev ? std::pow(c->opt.eps_a / (double)t, c->opt.eps_b) : c->opt.eps;
    N.eps = (float)eps;
    N.sd = (float)std::sqrt(2.0 * eps);
    const int64_t np = c->part_n[part];
    N.S = c->opt.scale_mode == PSGLD_SCALE_B ? (float)c->B
                                             : (np > 0 ? (float)((double)c->N / (double)np) : 0.f);
    N.mirror = c->prior.kind == PSGLD_PRIOR_EXPONENTIAL;
    uint32_t k0 = (uint32_t)c->opt.seed, k1 = (uint32_t)(c->opt.seed >> 32);
    for (int r = 0; r < 10; ++r) {   // Weyl key schedule of Philox4x32
        N.rk0[r] = k0;
        N.rk1[r] = k1;
        k0 += 0x9E3779B9u;
        k1 += 0xBB67AE85u;
    }
}

// Update parameters of iteration t (part `part`) for dense context c.  With
// t_dev the update kernel reads t from *t_dev + t_add.
static void fill_params(psgld_ctx *c, int part, int64_t t, const int64_t *t_dev, int64_t t_add, UpdParams &UP)
{
    const bool upd[2] = {!c->opt.freeze_W, !c->opt.freeze_H};
    UP = UpdParams{};
    for (int s = 0; s < 2; ++s) {
        UpdSide &Us = UP.side[s];
        const int64_t n_rows = s == 0 ? c->I : c->J;
        Us.X_cur = s == 0 ? c->W[c->wcur] : c->Ht[c->hcur];
        Us.X_next = s == 0 ? c->W[c->wcur ^ 1] : c->Ht[c->hcur ^ 1];
        Us.Gin = c->G + (s == 0 ? 0 : c->I * c->ldk);
        Us.gparts = 1;
        if (c->dense_kind == 1 && s == 1 && c->mtiles > 1) {
            Us.Gin = c->hpart;
            Us.gparts = c->mtiles;
            Us.gstride = c->J * c->ldk;
        }
        Us.n_rows = n_rows;
        if (c->dense_kind == 2) {
            Us.sh = s == 0 ? c->Wsh : c->Hsh;
            Us.sh_tiles = 2 * (s == 0 ? c->mt_max : c->nt_max);
        }
        Us.items = upd[s] ? n_rows * c->ngroups : 0;
        if (c->prior.kind == PSGLD_PRIOR_EXPONENTIAL) {
            Us.prior_a = (float)-(s == 0 ? c->prior.lambda_w : c->prior.lambda_h);
        } else {
            const double sg = s == 0 ? c->prior.sigma_w : c->prior.sigma_h;
            Us.prior_b = (float)(-1.0 / (sg * sg));
        }
    }
    fill_noise(c, part, t, t_dev, t_add, UP.noise);
    UP.K = c->K;
    UP.ldk = c->ldk;
    UP.ngroups = c->ngroups;
    const int64_t max_items = std::max(UP.side[0].items, UP.side[1].items);
    UP.div_magic = (max_items * c->ngroups < (1ll << 32))
                       ? (uint32_t)(((1ull << 32) + c->ngroups - 1) / c->ngroups)
                       : 0u;
    UP.B = c->B;
    UP.sh_kp = c->KP;
    // 32-bit arithmetic: items, factor rows, every partial gradient array and
    // the BF16 shadows within 2^31
    const int64_t lim = (1ll << 31) - 1;
    const int64_t sh_elems = c->dense_kind == 2
        ? (int64_t)c->B * 2 * std::max<int64_t>(c->mt_max, c->nt_max) * 64 * c->KP : 0;
    UP.small = UP.side[0].items + UP.side[1].items <= lim && std::max(c->I, c->J) * c->ldk <= lim &&
               (int64_t)std::max(1, c->mtiles) * c->J * c->ldk <= lim && sh_elems <= lim;
}

psgld_status launch_part_step(psgld_ctx *c, int64_t t, const int64_t *t_dev, int64_t t_add,
                              cudaStream_t st)
{
    const int B = c->B;
    const int part = part_of_iteration(c, t);
    const bool upd[2] = {!c->opt.freeze_W, !c->opt.freeze_H};
    // Inside a stream capture the records must be external, so that they
    // become event-record nodes of the graph (a plain record would only
    // become a dependency edge); outside a capture they are plain records.
    const bool prof = c->opt.profile && (int)c->ev_start.size() == B;
    unsigned rec_flags = cudaEventRecordDefault;
    if (prof) {
        cudaStreamCaptureStatus cap = cudaStreamCaptureStatusNone;
        PSGLD_CK(c, cudaStreamIsCapturing(st, &cap));
        if (cap == cudaStreamCaptureStatusActive) rec_flags = cudaEventRecordExternal;
        PSGLD_CK(c, cudaEventRecordWithFlags(c->ev_start[part], st, rec_flags));
    }
    if (!c->dense) {
        if (c->units) {
            const psgld_status rs = launch_units(c, part, t, t_dev, t_add, st, prof ? c->ev_mid[part] : nullptr, rec_flags);
            if (rs != PSGLD_OK) return rs;
        } else {
            const psgld_status rs = launch_rows(c, part, t, t_dev, t_add, st);
            if (rs != PSGLD_OK) return rs;
            // gradient and update are one launch, profiled as the gradient's
            if (prof) PSGLD_CK(c, cudaEventRecordWithFlags(c->ev_mid[part], st, rec_flags));
        }
    } else {
        UpdParams UP;
        fill_params(c, part, t, t_dev, t_add, UP);
        if (upd[0] || upd[1]) {
            const psgld_status ds = launch_dense_grad(c, part, st);
            if (ds != PSGLD_OK) return ds;
        }
        PSGLD_CK(c, cudaGetLastError());
        if (prof) PSGLD_CK(c, cudaEventRecordWithFlags(c->ev_mid[part], st, rec_flags));
        const int64_t items = UP.side[0].items + UP.side[1].items;
        const int grid = (int)std::min<int64_t>((items + kThreads - 1) / kThreads, 152 * 16);
        if (grid > 0) {
            PSGLD_CK(c, launch_early(!prof, UP.small ? update_kernel_dense32 : update_kernel, (unsigned)grid, kThreads,
                                     0, st, UP));
        }
    }
    PSGLD_CK(c, cudaGetLastError());
    if (prof) {
        PSGLD_CK(c, cudaEventRecordWithFlags(c->ev_end[part], st, rec_flags));
        c->ev_pending[part] = 1;
    }
    if (upd[0]) c->wcur ^= 1;
    if (upd[1]) c->hcur ^= 1;
    return PSGLD_OK;
}

namespace {

// ---- many contexts in one update launch ------------------------------------

// Block b takes a contiguous run of the items of all contexts, so that it
// looks a context up once and then steps from one to the next (256 chains of
// 513 x 200-5000, K = 32: a launch 115 to 91 us, with 32-bit index arithmetic
// where a context's arrays allow it).
__global__ void __launch_bounds__(kThreads, 4)
update_batch_kernel(const UpdParams *__restrict__ Ps, const int64_t *__restrict__ item_start, int n)
{
    dev::wait_prior();
    dev::let_next();
    const int64_t total = __ldg(item_start + n);
    const int64_t per = ((total + gridDim.x - 1) / gridDim.x + kThreads - 1) / kThreads * kThreads;
    const int64_t from = blockIdx.x * per, to = from + per < total ? from + per : total;
    if (from >= to) return;
    int ci;
    {
        int lo = 0, hi = n - 1;   // last i with item_start[i] <= from
        while (lo < hi) {
            const int mid = (lo + hi + 1) >> 1;
            if (__ldg(item_start + mid) <= from) lo = mid; else hi = mid - 1;
        }
        ci = lo;
    }
    for (int64_t begin = from; begin < to; ++ci) {   // one context's part of the run
        const int64_t first = __ldg(item_start + ci), next = __ldg(item_start + ci + 1);
        const int64_t end = next < to ? next : to;
        const UpdParams &P = Ps[ci];
        float eps, sd;
        const int64_t t = read_step(P, eps, sd);
        const uint32_t t_lo = (uint32_t)(uint64_t)t, t_hi = (uint32_t)((uint64_t)t >> 32);
        const int64_t n0 = P.side[0].items;
        if (P.small) {
            const uint32_t w = (uint32_t)n0;
            for (uint32_t a = (uint32_t)(begin - first) + threadIdx.x; a < (uint32_t)(end - first); a += kThreads) {
                if (a < w) update_item_dense32<0>(P, a, eps, sd, t_lo, t_hi);
                else update_item_dense32<1>(P, a - w, eps, sd, t_lo, t_hi);
            }
        } else {
            for (int64_t a = begin - first + threadIdx.x; a < end - first; a += kThreads) {
                if (a < n0) update_item<0>(P, a, eps, sd, t_lo, t_hi);
                else update_item<1>(P, a - n0, eps, sd, t_lo, t_hi);
            }
        }
        begin = end;
    }
}

}  // namespace

size_t upd_param_bytes() { return sizeof(UpdParams); }

int64_t fill_upd_param(psgld_ctx *c, int part, const int64_t *t_dev, int64_t t_add, void *dst)
{
    UpdParams UP;
    fill_params(c, part, t_add, t_dev, t_add, UP);
    UP.noise.eps_tab = nullptr;   // the batch's launches have no table: eps_t from t
    UP.eps_poly = c->opt.eps_mode == PSGLD_EPS_POLY;
    UP.eps_a = c->opt.eps_a;
    UP.eps_b = c->opt.eps_b;
    std::memcpy(dst, &UP, sizeof UP);
    return UP.side[0].items + UP.side[1].items;
}

psgld_status launch_update_batch(psgld_ctx *c0, const void *params, const int64_t *item_start, int n,
                                 int64_t total_items, bool early, cudaStream_t st)
{
    const int64_t cap = c0->opt.batch_update_blocks > 0 ? c0->opt.batch_update_blocks : 152 * 16;
    const int grid = (int)std::min<int64_t>((total_items + kThreads - 1) / kThreads, cap);
    if (grid > 0)
        PSGLD_CK(c0, launch_early(early, update_batch_kernel, (unsigned)grid, kThreads, 0, st,
                                  static_cast<const UpdParams *>(params), item_start, n));
    return PSGLD_OK;
}

}  // namespace psgld
