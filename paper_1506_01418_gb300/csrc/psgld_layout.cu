// psgld_layout.cu -- device construction of the part-major layouts.
//
// Blocks and parts (Definitions 1 and 2 of the paper): row piece r of [I] is
// [floor(r I / B), floor((r+1) I / B)); at iteration t the part pairs row
// piece r with column piece (r + s) mod B, s = (t-1) mod B.  So an observed
// entry (i, j) belongs to the part s = (piece(j) - piece(i)) mod B, and the
// layouts group entries by part:
//   A side: key (s*I + i, j)  -> CSR of every part over all I rows
//   B side: key (s*J + j, i)  -> CSC of every part over all J columns
// Both are produced by a stable LSD radix sort written here (8-bit digits,
// per-tile histograms, a global exclusive scan and a stable scatter whose
// in-tile ranks come from warp match/ballot), so the order is exact and
// repeatable.  What is sorted are whole entries (a 32-bit key, the other
// index, the value), so the last pass writes the layout itself.  The A side
// of entries that come in row-major order needs the parts' digits alone
// (stable: rows and columns stay in order within a part), one pass for up to
// 256 parts; other entries take the columns' digits, then those of s*I + i.
// The B side starts from the A side, whose parts hold their rows in order, so
// the digits of s*J + j are enough.  10^7 entries, 70000 x 10000, B = 32: 4
// passes, where sorting 64-bit (part, row, column) keys with a permutation
// took 5 for each side and gathered the entries through it afterwards; load,
// factors and a part-step 3.99 to 1.54 ms.
// The A side's entries also keep their row of W, for the reductions over all
// entries, and both sides list, per part, the rows with many entries, which
// the part-step gives more lanes.
#include <algorithm>
#include <utility>

#include "psgld_internal.cuh"
#include "psgld_slots.cuh"

namespace psgld {

int bits_for(uint64_t n_values)
{
    int b = 0;
    while (b < 64 && (n_values > (1ull << b))) ++b;
    return b;
}

namespace {

constexpr int kScanThreads = 256;
constexpr int kScanItems = 16;
constexpr int kScanTile = kScanThreads * kScanItems;

// Exclusive scan of one tile held in shared memory (n <= kScanTile valid
// values, the rest zero); returns the tile total to thread 0.
__device__ uint32_t block_exclusive_scan(uint32_t *sm, int n)
{
    __shared__ uint32_t warp_tot[kScanThreads / 32];
    const int tid = threadIdx.x;
    uint32_t v[kScanItems];
    uint32_t run = 0;
#pragma unroll
    for (int k = 0; k < kScanItems; ++k) {
        const int a = tid * kScanItems + k;
        v[k] = a < n ? sm[a] : 0u;
        run += v[k];
    }
    // inclusive warp scan of the per-thread totals
    const int lane = tid & 31, warp = tid >> 5;
    uint32_t inc = run;
#pragma unroll
    for (int o = 1; o < 32; o <<= 1) {
        uint32_t y = __shfl_up_sync(0xffffffffu, inc, o);
        if (lane >= o) inc += y;
    }
    if (lane == 31) warp_tot[warp] = inc;
    __syncthreads();
    if (warp == 0) {
        uint32_t w = lane < kScanThreads / 32 ? warp_tot[lane] : 0u;
        uint32_t wi = w;
#pragma unroll
        for (int o = 1; o < 32; o <<= 1) {
            uint32_t y = __shfl_up_sync(0xffffffffu, wi, o);
            if (lane >= o) wi += y;
        }
        if (lane < kScanThreads / 32) warp_tot[lane] = wi - w;  // exclusive
    }
    __syncthreads();
    uint32_t base = warp_tot[warp] + inc - run;
    uint32_t total = 0;
    if (tid == kScanThreads - 1) total = base + run;
#pragma unroll
    for (int k = 0; k < kScanItems; ++k) {
        const int a = tid * kScanItems + k;
        if (a < n) sm[a] = base;
        base += v[k];
    }
    __syncthreads();
    return total;
}

__global__ void scan_tile_sums(const uint32_t *__restrict__ in, int64_t n,
                               uint32_t *__restrict__ sums)
{
    const int64_t base = (int64_t)blockIdx.x * kScanTile;
    uint32_t s = 0;
    for (int k = threadIdx.x; k < kScanTile; k += kScanThreads)
        if (base + k < n) s += in[base + k];
    for (int o = 16; o > 0; o >>= 1) s += __shfl_xor_sync(0xffffffffu, s, o);
    __shared__ uint32_t ws[kScanThreads / 32];
    if ((threadIdx.x & 31) == 0) ws[threadIdx.x >> 5] = s;
    __syncthreads();
    if (threadIdx.x == 0) {
        uint32_t t = 0;
        for (int w = 0; w < kScanThreads / 32; ++w) t += ws[w];
        sums[blockIdx.x] = t;
    }
}

// One CTA scans in -> out (exclusive; in place where they are the same), tile
// by tile with a carry.
__global__ void scan_single(const uint32_t *in, int64_t n, uint32_t *out, uint32_t *total)
{
    __shared__ uint32_t sm[kScanTile];
    __shared__ uint32_t carry;
    if (threadIdx.x == 0) carry = 0;
    __syncthreads();
    for (int64_t base = 0; base < n; base += kScanTile) {
        const int m = (int)(n - base < kScanTile ? n - base : kScanTile);
        for (int k = threadIdx.x; k < kScanTile; k += kScanThreads)
            sm[k] = k < m ? in[base + k] : 0u;
        __syncthreads();
        uint32_t t = block_exclusive_scan(sm, m);
        const uint32_t cbase = carry;
        for (int k = threadIdx.x; k < m; k += kScanThreads) out[base + k] = sm[k] + cbase;
        __syncthreads();
        if (threadIdx.x == kScanThreads - 1) carry = cbase + t;
        __syncthreads();
    }
    if (threadIdx.x == 0 && total) *total = carry;
}

__global__ void scan_tiles(const uint32_t *__restrict__ in, int64_t n,
                           const uint32_t *__restrict__ sums, uint32_t *__restrict__ out)
{
    __shared__ uint32_t sm[kScanTile];
    const int64_t base = (int64_t)blockIdx.x * kScanTile;
    const int m = (int)(n - base < kScanTile ? n - base : kScanTile);
    for (int k = threadIdx.x; k < kScanTile; k += kScanThreads)
        sm[k] = k < m ? in[base + k] : 0u;
    __syncthreads();
    block_exclusive_scan(sm, m);
    const uint32_t off = sums[blockIdx.x];
    for (int k = threadIdx.x; k < m; k += kScanThreads) out[base + k] = sm[k] + off;
}

// ---- radix sort -----------------------------------------------------------

constexpr int kSortThreads = 256;
constexpr int kSortItems = 16;
constexpr int kSortTile = kSortThreads * kSortItems;  // 4096 entries per CTA
constexpr int kSortWarps = kSortThreads / 32;

// Entries as three arrays: key, other index, value.
struct Entries {
    const uint32_t *key, *other;
    const float *val;
};

// Digit of an entry: 8 bits at `shift` of its key divided by `div`, or
// (by_other) of its other index.
struct Digit {
    uint32_t div;
    int shift, by_other;

    __device__ __forceinline__ uint32_t of(uint32_t key, uint32_t other) const
    {
        const uint32_t x = by_other ? other : div > 1 ? key / div : key;
        return (x >> shift) & 255u;
    }
};

__global__ void radix_hist(const Entries in, int64_t n, const Digit D, uint32_t *__restrict__ hist, int64_t ntiles)
{
    __shared__ uint32_t h[256];
    h[threadIdx.x] = 0;
    __syncthreads();
    const int64_t base = (int64_t)blockIdx.x * kSortTile;
    const uint32_t *src = D.by_other ? in.other : in.key;
    for (int k = threadIdx.x; k < kSortTile; k += kSortThreads) {
        const bool ok = base + k < n;
        const uint32_t x = ok ? __ldg(src + base + k) : 0u;
        const uint32_t d = ok ? D.of(x, x) : 256u;
        // equal digits of a warp count once (runs of one part or of one row's
        // high digit would serialise on one counter)
        const unsigned peers = __match_any_sync(0xffffffffu, d);
        if (ok && (threadIdx.x & 31) == __ffs(peers) - 1) atomicAdd(&h[d], (uint32_t)__popc(peers));
    }
    __syncthreads();
    hist[(int64_t)threadIdx.x * ntiles + blockIdx.x] = h[threadIdx.x];
}

// Stable scatter.  Warp w of the tile owns positions [w*512, (w+1)*512);
// item m of lane l is position w*512 + m*32 + l, so (w, m, l) order is
// position order.  Ranks among equal digits come from __match_any_sync.
__global__ void __launch_bounds__(kSortThreads)
radix_scatter(const Entries in, int64_t n, const Digit D, const uint32_t *__restrict__ offs, int64_t ntiles,
              uint32_t *__restrict__ key_out, uint32_t *__restrict__ other_out, float *__restrict__ val_out)
{
    __shared__ uint32_t wcnt[kSortWarps][256];
    const int lane = threadIdx.x & 31, warp = threadIdx.x >> 5;
    for (int d = threadIdx.x; d < kSortWarps * 256; d += kSortThreads) (&wcnt[0][0])[d] = 0;
    __syncthreads();
    const int64_t base = (int64_t)blockIdx.x * kSortTile + warp * (32 * kSortItems);
    const uint32_t lt = (1u << lane) - 1u;
    uint32_t key[kSortItems], other[kSortItems], at[kSortItems];   // at: rank << 9 | digit
#pragma unroll
    for (int m = 0; m < kSortItems; ++m) {
        const int64_t pos = base + m * 32 + lane;
        key[m] = pos < n ? __ldg(in.key + pos) : 0u;
        other[m] = pos < n ? __ldg(in.other + pos) : 0u;
    }
#pragma unroll
    for (int m = 0; m < kSortItems; ++m) {
        const bool ok = base + m * 32 + lane < n;
        const uint32_t d = ok ? D.of(key[m], other[m]) : 256u;
        const unsigned peers = __match_any_sync(0xffffffffu, d);
        const uint32_t before = ok ? wcnt[warp][d] : 0u;
        at[m] = ((before + __popc(peers & lt)) << 9) | d;
        __syncwarp();
        if (ok && (peers & lt) == 0) wcnt[warp][d] = before + __popc(peers);
        __syncwarp();
    }
    __syncthreads();
    {   // per digit (one a thread): where each warp's entries go
        const int d = threadIdx.x;
        uint32_t run = offs[(int64_t)d * ntiles + blockIdx.x];
        for (int w = 0; w < kSortWarps; ++w) {
            const uint32_t c = wcnt[w][d];
            wcnt[w][d] = run;
            run += c;
        }
    }
    __syncthreads();
#pragma unroll
    for (int m = 0; m < kSortItems; ++m) {
        const uint32_t d = at[m] & 511u;
        if (d < 256u) {
            const uint32_t dst = wcnt[warp][d] + (at[m] >> 9);
            key_out[dst] = key[m];
            other_out[dst] = other[m];
            val_out[dst] = __ldg(in.val + base + m * 32 + lane);
        }
    }
}

// ---- layout kernels ---------------------------------------------------------

// largest r with floor(r n / B) <= x; B n < 2^31 (checked at create)
__device__ __forceinline__ uint32_t piece_of(uint32_t x, uint32_t n, uint32_t B) { return ((x + 1u) * B - 1u) / n; }

// Checks the entries (flag: 1 index out of range, 2 value, 8 not in strict
// row-major order) and writes their slots of the A side, s*I + i.
__global__ void validate_and_key(int64_t nnz, const int32_t *__restrict__ ii, const int32_t *__restrict__ jj,
                                 const float *__restrict__ vv, uint32_t I, uint32_t J, uint32_t B, int nonneg,
                                 uint32_t *__restrict__ key, int *flag)
{
    int bad = 0;
    for (int64_t e = blockIdx.x * (int64_t)blockDim.x + threadIdx.x; e < nnz;
         e += (int64_t)gridDim.x * blockDim.x) {
        const uint32_t i = (uint32_t)ii[e], j = (uint32_t)jj[e];
        const float v = vv[e];
        if (i >= I || j >= J) { bad |= 1; continue; }
        if (!isfinite(v) || (nonneg && v < 0.0f)) bad |= 2;
        if (e > 0) {
            const uint32_t ip = (uint32_t)ii[e - 1], jp = (uint32_t)jj[e - 1];
            if (!(ip < i || (ip == i && jp < j))) bad |= 8;
        }
        const uint32_t rp = piece_of(i, I, B), cp = piece_of(j, J, B);
        key[e] = (cp >= rp ? cp - rp : cp + B - rp) * I + i;
    }
    bad = __reduce_or_sync(0xffffffffu, bad);
    if (bad && (threadIdx.x & 31) == 0) atomicOr(flag, bad);
}

// The B side's slots s*J + j and rows i from the A side's order.
__global__ void key_columns(int64_t nnz, const uint32_t *__restrict__ keyA, const uint32_t *__restrict__ jA, uint32_t I,
                            uint32_t J, uint32_t *__restrict__ keyB, uint32_t *__restrict__ iB)
{
    for (int64_t e = blockIdx.x * (int64_t)blockDim.x + threadIdx.x; e < nnz;
         e += (int64_t)gridDim.x * blockDim.x) {
        const uint32_t k = keyA[e], s = k / I;
        keyB[e] = s * J + jA[e];
        iB[e] = k - s * I;
    }
}

// The slots' first entries; duplicates flagged (4); the entries' own rows.
__global__ void finish_side(int64_t nnz, const uint32_t *__restrict__ key, const uint32_t *__restrict__ other,
                            uint32_t nslots, uint32_t n_rows, int32_t *__restrict__ own, int32_t *__restrict__ ptr,
                            int *flag)
{
    for (int64_t p = blockIdx.x * (int64_t)blockDim.x + threadIdx.x; p <= nnz;
         p += (int64_t)gridDim.x * blockDim.x) {
        const uint32_t slot = p < nnz ? key[p] : nslots;
        const uint32_t from = p > 0 ? key[p - 1] + 1u : 0u;
        for (uint32_t s = from; s <= slot; ++s) ptr[s] = (int32_t)p;
        if (p < nnz) {
            if (own) own[p] = (int32_t)(slot % n_rows);
            if (p > 0 && from == slot + 1u && other[p] == other[p - 1]) atomicOr(flag, 4);
        }
    }
}

// Per slot (row of a part): is it a mid row (heavy = 0), or how many chunks
// has it as a heavy one
__global__ void count_rows(const int32_t *__restrict__ ptr, int64_t nslots, int heavy, uint32_t light,
                           uint32_t *__restrict__ out)
{
    for (int64_t s = blockIdx.x * (int64_t)blockDim.x + threadIdx.x; s < nslots;
         s += (int64_t)gridDim.x * blockDim.x) {
        const uint32_t n = (uint32_t)(ptr[s + 1] - ptr[s]);
        out[s] = heavy ? (n > kMidRow ? (n + kChunk - 1) / kChunk : 0u) : (n > light && n <= kMidRow ? 1u : 0u);
    }
}

// The mid rows, or the heavy rows' chunks, in slot order (pos: exclusive
// scan of count_rows).
__global__ void list_rows(const uint32_t *__restrict__ pos, const int32_t *__restrict__ ptr, int64_t nslots,
                          uint32_t n_rows, int4 *__restrict__ list)
{
    for (int64_t s = blockIdx.x * (int64_t)blockDim.x + threadIdx.x; s < nslots;
         s += (int64_t)gridDim.x * blockDim.x) {
        const uint32_t a = pos[s], b = pos[s + 1];
        if (b > a) {
            const int row = (int)((uint32_t)s % n_rows), first = ptr[s], n = ptr[s + 1] - first;
            for (uint32_t k = a; k < b; ++k) list[k] = make_int4(row, first, n, (int)(k - a));
        }
    }
}

// out[s] = x[s n_rows], s = 0 .. B: where each part begins
__global__ void gather_starts(const uint32_t *__restrict__ x, int64_t n_rows, int B, int64_t *__restrict__ out)
{
    for (int s = threadIdx.x; s <= B; s += blockDim.x) out[s] = x[(int64_t)s * n_rows];
}

int grid_for(int64_t n, int threads)
{
    int64_t g = (n + threads - 1) / threads;
    return (int)std::max<int64_t>(1, std::min<int64_t>(g, 152 * 32));
}

// Several arrays in one allocation: sizes first, then the addresses.
struct Arena {
    size_t bytes = 0;
    std::vector<std::pair<void **, size_t>> parts;

    template <typename T>
    void add(T **p, int64_t n)
    {
        parts.emplace_back(reinterpret_cast<void **>(p), bytes);
        bytes += (sizeof(T) * (size_t)std::max<int64_t>(n, 1) + 255) & ~size_t(255);
    }
    void place(void *base) const
    {
        for (const auto &q : parts) *q.first = static_cast<unsigned char *>(base) + q.second;
    }
};

// Exclusive scan of n uint32 values (in -> out, out has n+1 entries; out[n]
// is the total).  tmp needs ceil(n / kScanTile) + 1 entries.  Up to four tiles
// one CTA in one launch: 21 255 entries of 6812 x 290, B = 10, load in 564 us,
// with three launches for every scan in 625.
psgld_status exclusive_scan(psgld_ctx *c, const uint32_t *in, uint32_t *out, int64_t n,
                            uint32_t *tmp, cudaStream_t st)
{
    const int64_t tiles = std::max<int64_t>(1, (n + kScanTile - 1) / kScanTile);
    if (tiles <= 4) {
        scan_single<<<1, kScanThreads, 0, st>>>(in, n, out, out + n);
        PSGLD_CK(c, cudaGetLastError());
        return PSGLD_OK;
    }
    scan_tile_sums<<<(unsigned)tiles, kScanThreads, 0, st>>>(in, n, tmp);
    scan_single<<<1, kScanThreads, 0, st>>>(tmp, tiles, tmp, out + n);
    scan_tiles<<<(unsigned)tiles, kScanThreads, 0, st>>>(in, n, tmp, out);
    PSGLD_CK(c, cudaGetLastError());
    return PSGLD_OK;
}

// The digits of one sort, lowest first.
std::vector<Digit> digits(uint32_t div, int bits, int by_other)
{
    std::vector<Digit> d;
    for (int shift = 0; shift < std::max(bits, 1); shift += 8) d.push_back({div, shift, by_other});
    return d;
}

// Sorts by the given digits: from `in` through the two scratch sets, the last
// pass's other index and value to `other_out` and `val_out`; returns the
// sorted keys in *key_out (one of the scratch arrays).
psgld_status radix_sort(psgld_ctx *c, Entries in, const std::vector<Digit> &ds, int64_t n, uint32_t *const key[2],
                        uint32_t *const other[2], float *const val[2], uint32_t *other_out, float *val_out,
                        uint32_t *hist, uint32_t *hist_scan, uint32_t *tmp, const uint32_t **key_out, cudaStream_t st)
{
    const int64_t ntiles = std::max<int64_t>(1, (n + kSortTile - 1) / kSortTile);
    int to = in.key == key[0] ? 1 : 0;
    for (size_t p = 0; p < ds.size(); ++p) {
        const bool end = p + 1 == ds.size();
        radix_hist<<<(unsigned)ntiles, kSortThreads, 0, st>>>(in, n, ds[p], hist, ntiles);
        psgld_status s = exclusive_scan(c, hist, hist_scan, 256 * ntiles, tmp, st);
        if (s != PSGLD_OK) return s;
        uint32_t *o = end ? other_out : other[to];
        float *v = end ? val_out : val[to];
        radix_scatter<<<(unsigned)ntiles, kSortThreads, 0, st>>>(in, n, ds[p], hist_scan, ntiles, key[to], o, v);
        PSGLD_CK(c, cudaGetLastError());
        in = {key[to], o, v};
        to ^= 1;
    }
    *key_out = in.key;
    return PSGLD_OK;
}

}  // namespace

void free_layout(psgld_ctx *c)
{
    // work that reads the layouts must be finished before they are handed back
    wait_enqueued(c);
    if (c->capture_stream) cudaStreamSynchronize(c->capture_stream);
    for (auto &sd : c->side) sd = SideLayout{};
    dev_free(c, c->layout_mem);
    dev_free(c, c->chunk_mem);
    c->layout_mem = c->chunk_mem = nullptr;
    c->layout_bytes = 0;
    dev_free(c, c->Vd);
    dev_free(c, c->hpart);
    dev_free(c, c->VA);
    dev_free(c, c->VB);
    dev_free(c, c->Et);
    dev_free(c, c->tsync);
    dev_free(c, c->Wsh);
    dev_free(c, c->Hsh);
    c->Vd = nullptr;
    c->hpart = nullptr;
    c->VA = c->VB = nullptr;
    c->Et = nullptr;
    c->tsync = nullptr;
    c->Wsh = c->Hsh = nullptr;
    c->dense_kind = 0;
    c->dense_fp8 = 0;
    c->dense = false;
    c->ldv = 0;
    c->mtiles = 0;
    c->units = false;
    c->has_data = false;
    c->N = 0;
    c->part_n.clear();
}

psgld_status build_layout(psgld_ctx *c, int64_t nnz, const int32_t *i_dev, const int32_t *j_dev,
                          const float *v_dev, cudaStream_t st)
{
    // the memory of the layout before stays when it fits this one
    void *kept = c->layout_mem;
    const size_t kept_bytes = c->layout_bytes;
    c->layout_mem = nullptr;
    free_layout(c);
    const int64_t I = c->I, J = c->J, n = nnz;
    const int B = c->B;
    c->light_row = light_row_for(I, J, c->ngroups);
    c->units = step_by_units(I, J, c->ngroups, n, B, c->opt.gather_bf16 != 0);
    if (c->units) {
        const psgld_status s = prepare_units(c);
        if (s != PSGLD_OK) { dev_free(c, kept, st); return s; }
    }

    const int64_t ntiles = std::max<int64_t>(1, (n + kSortTile - 1) / kSortTile);
    const int64_t nslots_max = (int64_t)B * std::max(I, J);
    const int64_t scan_n = std::max<int64_t>(256 * ntiles + 1, nslots_max + 1);
    const int64_t tmp_n = (scan_n + kScanTile - 1) / kScanTile + 2;
    uint32_t *key[2], *other[2], *hist, *hscan, *tmp;
    float *val[2];
    int64_t *offs_dev;   // starts of the parts' entries, mid rows and chunks, per side
    Arena scratch, keep;
    for (int b = 0; b < 2; ++b) {
        scratch.add(&key[b], n);
        scratch.add(&other[b], n);
        scratch.add(&val[b], n);
    }
    scratch.add(&hist, scan_n);
    scratch.add(&hscan, scan_n + 1);
    scratch.add(&tmp, tmp_n);
    scratch.add(&offs_dev, 6 * ((int64_t)B + 1));
    for (int side = 0; side < 2; ++side) {
        SideLayout &sd = c->side[side];
        const int64_t nslots = (int64_t)B * (side == 0 ? I : J);
        keep.add(&sd.ptr, nslots + 1);
        keep.add(&sd.idx, n);
        keep.add(&sd.val, n);
        if (side == 0 || c->units) keep.add(&sd.own, n);
        keep.add(&sd.mid, std::min(n / (c->light_row + 1), nslots));
        keep.add(&sd.heavy, max_chunks(n));
    }
    if (kept && (kept_bytes < keep.bytes || kept_bytes > 2 * keep.bytes)) {
        dev_free(c, kept, st);
        kept = nullptr;
    }
    void *scratch_mem = dev_alloc(c, scratch.bytes, st);
    if (!scratch_mem && kept) {   // as large as twice this layout: make room
        dev_free(c, kept, st);
        kept = nullptr;
        scratch_mem = dev_alloc(c, scratch.bytes, st);
    }
    c->layout_mem = kept ? kept : dev_alloc(c, keep.bytes, st);
    c->layout_bytes = kept ? kept_bytes : keep.bytes;
    auto cleanup = [&]() {
        cudaStreamSynchronize(st);   // the scratch is in use by work on st
        dev_free(c, scratch_mem, st);
        scratch_mem = nullptr;
    };
    auto give_up = [&](psgld_status s) {
        cleanup();
        free_layout(c);
        return s;
    };
    if (!scratch_mem || !c->layout_mem)
        return give_up(fail(c, PSGLD_ERR_OOM, "device allocation of " + std::to_string(scratch.bytes + keep.bytes) +
                                                  " bytes for the layout failed"));
    scratch.place(scratch_mem);
    keep.place(c->layout_mem);

    cudaError_t e = cudaMemsetAsync(c->flag, 0, sizeof(int), st);
    if (n > 0)
        validate_and_key<<<grid_for(n, 256), 256, 0, st>>>(n, i_dev, j_dev, v_dev, (uint32_t)I, (uint32_t)J, (uint32_t)B,
                                                           c->prior.kind == PSGLD_PRIOR_EXPONENTIAL, key[0], c->flag);
    if (e == cudaSuccess) e = cudaGetLastError();
    int hflag = 0;
    if (e == cudaSuccess) e = cudaMemcpyAsync(&hflag, c->flag, sizeof(int), cudaMemcpyDeviceToHost, st);
    if (e == cudaSuccess) e = cudaStreamSynchronize(st);
    if (e != cudaSuccess) return give_up(cuda_fail(c, e, "layout: entry checks"));
    if (hflag & 1) return give_up(fail(c, PSGLD_ERR_ARG, "entry index out of range"));
    if (hflag & 2) return give_up(fail(c, PSGLD_ERR_ARG, "entry value not finite, or negative in a non-negative model"));

    const uint32_t *sorted = key[0];
    for (int side = 0; side < 2; ++side) {
        SideLayout &sd = c->side[side];
        const int64_t n_rows = side == 0 ? I : J;
        const int64_t nslots = (int64_t)B * n_rows;
        if (n > 0) {
            Entries in;
            std::vector<Digit> ds;
            if (side == 0) {
                in = {key[0], reinterpret_cast<const uint32_t *>(j_dev), v_dev};
                if (!(hflag & 8)) {
                    ds = digits((uint32_t)I, bits_for((uint64_t)B), 0);
                } else {
                    ds = digits(1, bits_for((uint64_t)J), 1);
                    for (const Digit &d : digits(1, bits_for((uint64_t)nslots), 0)) ds.push_back(d);
                }
            } else {
                // the A side's sorted keys are in one of the two key arrays
                uint32_t *kb = sorted == key[0] ? key[1] : key[0];
                key_columns<<<grid_for(n, 256), 256, 0, st>>>(n, sorted, reinterpret_cast<const uint32_t *>(c->side[0].idx),
                                                              (uint32_t)I, (uint32_t)J, kb, kb == key[0] ? other[0] : other[1]);
                in = {kb, kb == key[0] ? other[0] : other[1], c->side[0].val};
                ds = digits(1, bits_for((uint64_t)nslots), 0);
            }
            const psgld_status s = radix_sort(c, in, ds, n, key, other, val, reinterpret_cast<uint32_t *>(sd.idx), sd.val,
                                              hist, hscan, tmp, &sorted, st);
            if (s != PSGLD_OK) return give_up(s);
        }
        finish_side<<<grid_for(n + 1, 256), 256, 0, st>>>(n, sorted, reinterpret_cast<const uint32_t *>(sd.idx),
                                                          (uint32_t)nslots, (uint32_t)n_rows, sd.own, sd.ptr, c->flag);
        int64_t *offs = offs_dev + 3 * side * ((int64_t)B + 1);
        gather_starts<<<1, 128, 0, st>>>(reinterpret_cast<const uint32_t *>(sd.ptr), n_rows, B, offs);
        for (int k = 0; k < 2; ++k) {
            count_rows<<<grid_for(nslots, 256), 256, 0, st>>>(sd.ptr, nslots, k, (uint32_t)c->light_row, hist);
            const psgld_status s = exclusive_scan(c, hist, hscan, nslots, tmp, st);
            if (s != PSGLD_OK) return give_up(s);
            list_rows<<<grid_for(nslots, 256), 256, 0, st>>>(hscan, sd.ptr, nslots, (uint32_t)n_rows,
                                                             k == 0 ? sd.mid : sd.heavy);
            gather_starts<<<1, 128, 0, st>>>(hscan, n_rows, B, offs + (k + 1) * (B + 1));
        }
        e = cudaGetLastError();
        if (e != cudaSuccess) return give_up(cuda_fail(c, e, "layout"));
    }
    std::vector<int64_t> h(6 * (size_t)(B + 1));
    e = cudaMemcpyAsync(h.data(), offs_dev, sizeof(int64_t) * h.size(), cudaMemcpyDeviceToHost, st);
    if (e == cudaSuccess) e = cudaMemcpyAsync(&hflag, c->flag, sizeof(int), cudaMemcpyDeviceToHost, st);
    if (e == cudaSuccess) e = cudaStreamSynchronize(st);
    if (e != cudaSuccess) return give_up(cuda_fail(c, e, "layout: offsets"));
    if (hflag & 4) return give_up(fail(c, PSGLD_ERR_ARG, "duplicate (i, j) entry"));
    cleanup();

    Arena chunk;
    int64_t chunks[2];
    for (int side = 0; side < 2; ++side) {
        SideLayout &sd = c->side[side];
        const int64_t *at = h.data() + 3 * side * (B + 1);
        if (side == 0) {
            c->part_n.resize(B);
            for (int p = 0; p < B; ++p) c->part_n[p] = at[p + 1] - at[p];
        }
        sd.part_first.assign(at, at + (B + 1));
        if (c->units) {
            int64_t floats = 0;
            for (int p = 0; p < B; ++p)
                floats = std::max(floats, slot_floats(at[p + 1] - at[p], unit_entries(c->ngroups), c->ldk));
            chunk.add(&sd.unit_sums, floats);
        }
        sd.mid_first.assign(at + (B + 1), at + 2 * (B + 1));
        sd.heavy_first.assign(at + 2 * (B + 1), at + 3 * (B + 1));
        chunks[side] = 0;
        for (int p = 0; p < B; ++p) chunks[side] = std::max(chunks[side], sd.heavy_first[p + 1] - sd.heavy_first[p]);
        if (chunks[side] > 0) {
            chunk.add(&sd.partial, chunks[side] * c->ldk);
            chunk.add(&sd.arrived, chunks[side]);
        }
    }
    if (chunk.bytes > 0) {
        c->chunk_mem = dev_alloc(c, chunk.bytes, st);
        if (!c->chunk_mem) return give_up(fail(c, PSGLD_ERR_OOM, "device allocation failed"));
        chunk.place(c->chunk_mem);
        for (int side = 0; side < 2; ++side)
            if (chunks[side] > 0) {
                e = cudaMemsetAsync(c->side[side].arrived, 0, sizeof(int) * (size_t)chunks[side], st);
                if (e != cudaSuccess) return give_up(cuda_fail(c, e, "memset"));
            }
    }
    c->N = n;
    c->has_data = true;
    return PSGLD_OK;
}

}  // namespace psgld
