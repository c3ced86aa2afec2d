// psgld_readout.cu -- posterior means and variances to host arrays.
//
// Mean and variance are formed on the device from the FP64 sums, a block of
// rows at a time, copied to pinned staging memory, and from there to the
// caller's arrays by several threads.  The caller's arrays are often new
// memory: copies straight into it fault from the device, 64 KB page by page
// (64 MB: 30 ms), and one thread alone spends most of its time getting pages
// (3.5 ms).  70000 x 10000, K = 50: 11.4 to 2.5 ms a read-back (before: the
// sums through staging arrays of their own, and the divisions on the host).
#include <algorithm>
#include <atomic>
#include <cmath>
#include <condition_variable>
#include <cstring>
#include <mutex>
#include <thread>

#include "psgld_internal.cuh"

namespace psgld {
namespace {

// Means (var = 0) or variances of `total` / K whole rows: rows of ldk sums
// to rows of K.
__global__ void moments_kernel(const double *__restrict__ s, const double *__restrict__ s2, int64_t total, int ldk,
                               int K, double n, int var, double *__restrict__ out)
{
    for (int64_t a = blockIdx.x * (int64_t)blockDim.x + threadIdx.x; a < total;
         a += (int64_t)gridDim.x * blockDim.x) {
        const int64_t r = a / K, at = r * ldk + (a - r * K);
        const double m = n > 0 ? s[at] / n : 0.0;
        out[a] = !var ? m : n > 0 ? fma(-m, m, s2[at] / n) : 0.0;
    }
}

constexpr size_t kHalf = 4 << 20;      // staging: two halves, one filled while the other is emptied
constexpr size_t kSlice = 256 << 10;   // bytes a thread copies at a time
// Up to this the sums are copied and divided on the host, one blocking copy at a
// time.  Moments of 0.05, 0.4, 0.8, 1.3, 1.6 MB, K = 16: 60, 96, 138, 191, 219 us
// (into new memory 104, 150, 201, 260, 303), through staging -, -, -, 196, 216
// (-, -, -, 243, 273).  Copied from the device straight to the caller's arrays
// 0.8 to 1 MB take 140 us, but 890 into new memory; four asynchronous copies and
// one wait instead of the blocking ones 66, 103, 139.
constexpr size_t kHost = 1536 << 10;
// bytes per helping thread: of 1.8 MB with seven 666 us, with none 229; of 8 MB
// 866, 776 with one, 897 with none; of 40 MB 1509, 3562 with none
constexpr int64_t kPerHelper = 4 << 20;
constexpr unsigned kThreads = 8;

// Staging areas of the process, at most kAreas (64 MB), one to a read-back
// while it lasts, given back with the last context.  A read-back that finds
// them all taken divides on the host.
constexpr int kAreas = 8;
std::mutex g_stage_mutex;
char *g_free[kAreas];
int g_n_free = 0, g_areas = 0, g_readers = 0;
int64_t g_contexts = 0;

class Staging {
public:
    // the area, if one is to be had, and how many read-backs there are now
    char *take(int *readers)
    {
        {
            std::lock_guard<std::mutex> l(g_stage_mutex);
            *readers = ++g_readers;
            reading_ = true;
            if (g_n_free > 0) return area_ = g_free[--g_n_free];
            if (g_areas == kAreas) return nullptr;
            ++g_areas;
        }
        if (cudaHostAlloc(reinterpret_cast<void **>(&area_), 2 * kHalf, cudaHostAllocPortable) != cudaSuccess) {
            cudaGetLastError();
            area_ = nullptr;
            std::lock_guard<std::mutex> l(g_stage_mutex);
            --g_areas;
        }
        return area_;
    }
    ~Staging()
    {
        if (!reading_) return;
        std::lock_guard<std::mutex> l(g_stage_mutex);
        --g_readers;
        if (area_) g_free[g_n_free++] = area_;
    }

private:
    char *area_ = nullptr;
    bool reading_ = false;
};

// Threads that copy slices beside the caller's, for one read-back.
class Crew {
public:
    explicit Crew(unsigned helpers)
    {
        try {
            for (unsigned k = 0; k < helpers; ++k) threads_.emplace_back([this] { serve(); });
        } catch (...) {   // as many as there are to be had
        }
    }
    ~Crew()
    {
        {
            std::lock_guard<std::mutex> l(m_);
            stop_ = true;
        }
        go_.notify_all();
        for (auto &t : threads_) t.join();
    }
    void copy(char *dst, const char *src, size_t bytes)
    {
        {
            std::lock_guard<std::mutex> l(m_);
            dst_ = dst;
            src_ = src;
            bytes_ = bytes;
            next_ = 0;
            busy_ = threads_.size();
            ++job_;
        }
        go_.notify_all();
        slices();
        std::unique_lock<std::mutex> l(m_);
        done_.wait(l, [this] { return busy_ == 0; });
    }

private:
    void slices()
    {
        for (size_t at; (at = next_.fetch_add(kSlice)) < bytes_;)
            std::memcpy(dst_ + at, src_ + at, std::min(kSlice, bytes_ - at));
    }
    void serve()
    {
        uint64_t seen = 0;
        std::unique_lock<std::mutex> l(m_);
        for (;;) {
            go_.wait(l, [&] { return stop_ || job_ != seen; });
            if (stop_) return;
            seen = job_;
            l.unlock();
            slices();
            l.lock();
            if (--busy_ == 0) done_.notify_one();
        }
    }
    std::vector<std::thread> threads_;
    std::mutex m_;
    std::condition_variable go_, done_;
    char *dst_ = nullptr;
    const char *src_ = nullptr;
    size_t bytes_ = 0, busy_ = 0;
    std::atomic<size_t> next_{0};
    uint64_t job_ = 0;
    bool stop_ = false;
};

struct Piece {
    int side, var;
    int64_t row, rows;
    double *out;
};

// G, dead between part-steps, holds the rows on their way out.
cudaError_t form(psgld_ctx *c, const Piece &p, cudaStream_t st)
{
    const Sums &S = p.side == 0 ? c->sW : c->sH;
    const int64_t n = p.rows * c->K;
    moments_kernel<<<(unsigned)std::min<int64_t>((n + 255) / 256, 152 * 16), 256, 0, st>>>(
        S.s + p.row * c->ldk, S.s2 + p.row * c->ldk, n, c->ldk, c->K, (double)c->n_samples, p.var,
        reinterpret_cast<double *>(c->G));
    return cudaGetLastError();
}

// The same moments, bit for bit, from the sums on the host.
psgld_status divide_on_host(psgld_ctx *c, double *const (&out)[2][2])
{
    const int64_t K = c->K, ldk = c->ldk;
    const double n = (double)c->n_samples;
    for (int side = 0; side < 2; ++side) {
        double *const mean = out[side][0], *const var = out[side][1];
        if (!mean && !var) continue;
        const Sums &S = side == 0 ? c->sW : c->sH;
        const int64_t rows = side == 0 ? c->I : c->J;
        std::vector<double> s((size_t)(rows * ldk)), s2(var ? s.size() : 0);
        PSGLD_CK(c, cudaMemcpy(s.data(), S.s, sizeof(double) * s.size(), cudaMemcpyDeviceToHost));
        if (var) PSGLD_CK(c, cudaMemcpy(s2.data(), S.s2, sizeof(double) * s2.size(), cudaMemcpyDeviceToHost));
        for (int64_t r = 0; r < rows; ++r)
            for (int64_t k = 0; k < K; ++k) {
                const int64_t at = r * ldk + k;
                const double m = n > 0 ? s[at] / n : 0.0;
                if (mean) mean[r * K + k] = m;
                if (var) var[r * K + k] = n > 0 ? std::fma(-m, m, s2[at] / n) : 0.0;
            }
    }
    return PSGLD_OK;
}

}  // namespace

void use_staging(int by)
{
    std::lock_guard<std::mutex> l(g_stage_mutex);
    g_contexts += by;
    if (g_contexts > 0) return;
    for (; g_n_free > 0; --g_areas) cudaFreeHost(g_free[--g_n_free]);
}

psgld_status read_moments(psgld_ctx *c, double *const (&out)[2][2])
{
    const size_t row = sizeof(double) * (size_t)c->K;
    int64_t total = 0;
    for (int side = 0; side < 2; ++side)
        for (int var = 0; var < 2; ++var)
            if (out[side][var]) total += (side == 0 ? c->I : c->J) * (int64_t)row;
    if (total <= (int64_t)kHost) return divide_on_host(c, out);
    Staging staging;
    int readers = 1;
    char *const area = staging.take(&readers);
    if (!area) return divide_on_host(c, out);
    const int64_t fit = (int64_t)(sizeof(float) * (size_t)((c->I + c->J) * c->ldk) / row);   // rows G holds
    const int64_t half = std::max<int64_t>(1, std::min<int64_t>(fit, kHalf / row));
    std::vector<Piece> pieces;
    for (int side = 0; side < 2; ++side)
        for (int var = 0; var < 2; ++var) {
            const int64_t rows = side == 0 ? c->I : c->J;
            if (!out[side][var]) continue;
            for (int64_t r = 0; r < rows; r += half)
                pieces.push_back({side, var, r, std::min(half, rows - r), out[side][var] + r * c->K});
        }
    cudaStream_t st = c->capture_stream;
    cudaEvent_t full[2] = {nullptr, nullptr};
    cudaError_t e = cudaSuccess;
    for (auto &ev : full)
        if (e == cudaSuccess) e = cudaEventCreateWithFlags(&ev, cudaEventDisableTiming);
    {
        // the host's cores among the read-backs under way
        const unsigned mine = std::max(1u, std::thread::hardware_concurrency() / (unsigned)readers);
        Crew crew((unsigned)std::min<int64_t>(std::min(kThreads, mine) - 1, total / kPerHelper));
        auto fetch = [&](size_t k) {
            e = form(c, pieces[k], st);
            if (e == cudaSuccess)
                e = cudaMemcpyAsync(area + (k & 1) * kHalf, c->G, row * (size_t)pieces[k].rows, cudaMemcpyDeviceToHost, st);
            if (e == cudaSuccess) e = cudaEventRecord(full[k & 1], st);
        };
        if (e == cudaSuccess) fetch(0);
        for (size_t k = 0; k < pieces.size() && e == cudaSuccess; ++k) {
            if (k + 1 < pieces.size()) fetch(k + 1);
            if (e == cudaSuccess) e = cudaEventSynchronize(full[k & 1]);
            if (e == cudaSuccess)
                crew.copy(reinterpret_cast<char *>(pieces[k].out), area + (k & 1) * kHalf, row * (size_t)pieces[k].rows);
        }
    }
    if (e != cudaSuccess) cudaStreamSynchronize(st);   // nothing in flight into the staging area
    for (auto &ev : full)
        if (ev) cudaEventDestroy(ev);
    if (e != cudaSuccess) return cuda_fail(c, e, "read-back of the posterior moments");
    return PSGLD_OK;
}

}  // namespace psgld
