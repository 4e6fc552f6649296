// Direct-sampling statistics of the drag (Sec. 3): the autocorrelation of the
// drag fluctuations and its correlation time (caption of Fig. pdf_drag), and
// the waiting-time return time r(a) of a level.  The ensemble's clones are
// independent trajectories; their drag series over [t0, t1) are pooled.  Means
// and variances are FP64 sums in a fixed order, the products of the
// autocorrelation exact integers (results do not depend on timing).
#include <algorithm>
#include <cmath>
#include <limits>
#include <type_traits>
#include <vector>

#include "internal.h"

namespace lbm {
namespace {

constexpr int kStatThreads = 256;

// fixed-order block sum of per-thread FP64 partials
__device__ double block_sum(double v, double* sh)
{
    sh[threadIdx.x] = v;
    __syncthreads();
    for (int s = kStatThreads / 2; s > 0; s >>= 1) {
        if ((int)threadIdx.x < s) sh[threadIdx.x] += sh[threadIdx.x + s];
        __syncthreads();
    }
    const double r = sh[0];
    __syncthreads();
    return r;
}

// The pooled series' moments, one block per clone: the sums; then, with the
// mean of all, the sums of squares and the largest fluctuation (stat[0 .. n):
// sums, [n .. 2n): squares, [2n .. 3n): largest |x|).  One block over the whole
// series with a 64-bit division per element took 1356 us (64 x 6500).
__global__ void drag_sum_kernel(const double* drag, int32_t max_steps, int32_t t0, int32_t len, double* stat)
{
    __shared__ double sh[kStatThreads];
    const double* row = drag + (int64_t)blockIdx.x * max_steps + t0;
    double s = 0.0;
    for (int t = threadIdx.x; t < len; t += kStatThreads) s += row[t];
    s = block_sum(s, sh);
    if (threadIdx.x == 0) stat[blockIdx.x] = s;
}

// the sum of n values by a whole block, in a fixed order
__device__ double sum_over(const double* v, int32_t n, double* sh)
{
    double s = 0.0;
    for (int i = threadIdx.x; i < n; i += kStatThreads) s += v[i];
    return block_sum(s, sh);
}

__global__ void drag_square_kernel(const double* drag, int32_t max_steps, int32_t n, int32_t t0, int32_t len,
                                   double* stat)
{
    __shared__ double sh[kStatThreads];
    const double mean = sum_over(stat, n, sh) / ((double)n * (double)len);
    const double* row = drag + (int64_t)blockIdx.x * max_steps + t0;
    double q = 0.0, top = 0.0;
    for (int t = threadIdx.x; t < len; t += kStatThreads) {
        const double x = row[t] - mean;
        q += x * x;
        top = fmax(top, fabs(x));
    }
    q = block_sum(q, sh);
    sh[threadIdx.x] = top;
    __syncthreads();
    for (int s = kStatThreads / 2; s > 0; s >>= 1) {
        if ((int)threadIdx.x < s) sh[threadIdx.x] = fmax(sh[threadIdx.x], sh[threadIdx.x + s]);
        __syncthreads();
    }
    if (threadIdx.x == 0) {
        stat[n + blockIdx.x] = q;
        stat[2 * n + blockIdx.x] = sh[0];
    }
}

// The autocorrelation's products in fixed point.  FP64 runs at two products a
// clock and SM on this GPU, 1.2 ms for the 7e8 products of 64 x 6500 steps and
// 2000 lags; 32-bit integer multiply-adds with 64-bit sums run 32 times as many.
// A fluctuation x is rounded to X = x 2^k with the largest below 2^54 (an error
// of 2^-55 of the largest, below the 2^-53 of an FP64 fluctuation of that size) and split
// into X = hi 2^28 + lo, |hi| <= 2^26 + 1, |lo| <= 2^27.  Every product is exact, and so
// is every sum after that, so the result does not depend on their order: 128
// bits would hold 2^19 products of the largest value (128 sine series of 20000
// steps sum to 2.2 x 2^127), so longer sums are kept in 160 bits, which hold 2^51.
constexpr int kLimb = 28;

// a sum of 128-bit integers v as that of v >> 32 and that of their low 32 bits
struct WideSum {
    __int128 high = 0;
    unsigned long long low = 0;
    __device__ void add(__int128 v)
    {
        high += v >> 32;
        low += (unsigned int)v;
    }
    __device__ void add(__int128 h, unsigned long long l)
    {
        high += h;
        low += l;
    }
    __device__ double value() const
    {
        __int128 h = high + (long long)(low >> 32);
        long long l = (long long)(low & 0xffffffffull);
        const bool negative = h < 0;  // then h 2^32 + l < 0: of the magnitude, no digits cancel
        if (negative) {
            h = -h;
            l = -l;
        }
        const double v = ((double)(long long)(h >> 64) * 0x1.0p64 + (double)(unsigned long long)h) * 0x1.0p32 + (double)l;
        return negative ? -v : v;
    }
};

// k of the quantisation; 0 for an all-zero or a non-finite series
__device__ int fixed_exponent(const double* stat, int32_t n, double* sh)
{
    double top = 0.0;
    for (int i = threadIdx.x; i < n; i += kStatThreads) top = fmax(top, stat[2 * n + i]);
    sh[threadIdx.x] = top;
    __syncthreads();
    for (int s = kStatThreads / 2; s > 0; s >>= 1) {
        if ((int)threadIdx.x < s) sh[threadIdx.x] = fmax(sh[threadIdx.x], sh[threadIdx.x + s]);
        __syncthreads();
    }
    top = sh[0];
    __syncthreads();
    return top > 0.0 && isfinite(top) ? 53 - ilogb(top) : 0;
}

// the limbs of every clone's fluctuations, [n][pitch] each, zeros past the series
__global__ void drag_limbs_kernel(const double* drag, int32_t max_steps, int32_t n, int32_t t0, int32_t len,
                                  const double* stat, int32_t pitch, int32_t* hi, int32_t* lo)
{
    __shared__ double sh[kStatThreads];
    const double mean = sum_over(stat, n, sh) / ((double)n * (double)len);
    const int k = fixed_exponent(stat, n, sh);
    const double s1 = scalbn(1.0, k / 2), s2 = scalbn(1.0, k - k / 2);
    const int64_t c = blockIdx.y;
    const int t = blockIdx.x * kStatThreads + threadIdx.x;
    if (t >= pitch) return;
    long long X = 0;
    if (t < len) X = __double2ll_rn((drag[c * max_steps + t0 + t] - mean) * s1 * s2);
    const long long h = (X + (1ll << (kLimb - 1))) >> kLimb;
    hi[c * pitch + t] = (int32_t)h;
    lo[c * pitch + t] = (int32_t)(X - (h << kLimb));
}

// Exact sums of products X(t) X(t + lag): a thread owns four consecutive lags
// and takes four times t at once from registers (16 products, 48 multiply-adds,
// for six 16-byte shared-memory loads; three multiply-adds a product instead of
// four through (hi + lo)(hi' + lo') - hi hi' - lo lo').  A block takes kCorrLags lags and walks
// its share of the (clone, kCorrTime steps) tasks; partial[split][lag].  A thread
// sums kCorrTasks tasks, 2^18 products, in 128 bits.  WIDE: it has more, and adds
// each kCorrTasks of them to its sum's halves in partial and low (the plain form
// stays beside it for its registers: 286 against 297 us, 64 x 6500 and 2000 lags).
constexpr int kCorrThreads = 128, kCorrLags = 4 * kCorrThreads, kCorrTime = 512, kCorrFlush = 128, kCorrTasks = 512;

template <bool WIDE>
__global__ void __launch_bounds__(kCorrThreads) autocorr_kernel(const int32_t* hi, const int32_t* lo, int32_t n,
                                                                int32_t len, int32_t pitch, int32_t n_lags,
                                                                __int128* partial, unsigned long long* low)
{
    constexpr int kWin = kCorrTime + kCorrLags + 4;
    __shared__ __align__(16) int32_t ah[kCorrTime], al[kCorrTime], as[kCorrTime], bh[kWin], bl[kWin], bs[kWin];
    const int chunks = (len + kCorrTime - 1) / kCorrTime, tasks = n * chunks;
    const int lag0 = blockIdx.x * kCorrLags, l0 = 4 * threadIdx.x;
    __int128 sum[4] = {0, 0, 0, 0};
    auto store = [&](bool more) {
#pragma unroll
        for (int j = 0; j < 4; ++j) {
            if (lag0 + l0 + j >= n_lags) continue;
            const int64_t i = (int64_t)blockIdx.y * n_lags + lag0 + l0 + j;
            if constexpr (WIDE) {
                WideSum w;
                if (more) w.add(partial[i], low[i]);
                w.add(sum[j]);
                partial[i] = w.high;
                low[i] = w.low;
                sum[j] = 0;
            } else {
                partial[i] = sum[j];
            }
        }
    };
    int done = 0;
    for (int task = blockIdx.y; task < tasks; task += gridDim.y) {
        if (WIDE && done++ % kCorrTasks == 0 && done > 1) store(done > kCorrTasks + 1);
        const int c = task / chunks, tb = (task - c * chunks) * kCorrTime;
        if (tb + lag0 >= len) continue;  // block-uniform: every product is past the series
        const int32_t *rh = hi + (int64_t)c * pitch, *rl = lo + (int64_t)c * pitch;
        __syncthreads();
        for (int i = threadIdx.x; i < kCorrTime; i += kCorrThreads) {
            ah[i] = rh[tb + i];  // the rows are zero up to their pitch
            al[i] = rl[tb + i];
            as[i] = ah[i] + al[i];
        }
        for (int i = threadIdx.x; i < kWin; i += kCorrThreads) {
            const int t = tb + lag0 + i;
            bh[i] = t < pitch ? rh[t] : 0;
            bl[i] = t < pitch ? rl[t] : 0;
            bs[i] = bh[i] + bl[i];
        }
        __syncthreads();
        for (int f = 0; f < kCorrTime; f += kCorrFlush) {
            // 128 products of each kind: below 2^60, 2^62 and 2^63
            long long hh[4] = {0, 0, 0, 0}, ll[4] = {0, 0, 0, 0}, ss[4] = {0, 0, 0, 0};
            auto at = [](const int32_t* v) { return *reinterpret_cast<const int4*>(v); };
            int4 wh = at(bh + f + l0), wl = at(bl + f + l0), ws = at(bs + f + l0);
#pragma unroll 2
            for (int t = f; t < f + kCorrFlush; t += 4) {
                const int4 vh = at(bh + t + 4 + l0), vl = at(bl + t + 4 + l0), vs = at(bs + t + 4 + l0);
                auto products = [](long long (&acc)[4], const int4& x, const int4& w, const int4& v) {
                    const int X[4] = {x.x, x.y, x.z, x.w}, Y[8] = {w.x, w.y, w.z, w.w, v.x, v.y, v.z, v.w};
#pragma unroll
                    for (int d = 0; d < 4; ++d)
#pragma unroll
                        for (int j = 0; j < 4; ++j) acc[j] += (long long)X[d] * Y[d + j];
                };
                products(hh, at(ah + t), wh, vh);
                products(ll, at(al + t), wl, vl);
                products(ss, at(as + t), ws, vs);
                wh = vh;
                wl = vl;
                ws = vs;
            }
#pragma unroll
            for (int j = 0; j < 4; ++j)
                sum[j] += ((__int128)hh[j] << (2 * kLimb)) + (((__int128)ss[j] - hh[j] - ll[j]) << kLimb) + (__int128)ll[j];
        }
    }
    store(done > kCorrTasks);
}

// C(lag) = sum of products / their number / variance; the first lag with C <= 0.
// A block takes 32 lags, each of its warps a part of the splits.
template <bool WIDE>
__global__ void __launch_bounds__(kStatThreads) autocorr_final_kernel(const __int128* partial,
                                                                      const unsigned long long* low, int32_t splits,
                                                                      int32_t n_lags, const double* stat, int32_t n,
                                                                      int32_t len, double* c, int32_t* first)
{
    __shared__ double sh[kStatThreads];
    const double var = sum_over(stat + n, n, sh) / ((double)n * (double)len);
    const int k = fixed_exponent(stat, n, sh);
    __shared__ __int128 part_h[kStatThreads / 32][32];
    __shared__ unsigned long long part_l[kStatThreads / 32][32];
    const int lane = threadIdx.x & 31, warp = threadIdx.x >> 5, lag = blockIdx.x * 32 + lane;
    WideSum s;
    if (lag < n_lags)
#pragma unroll 4
        for (int i = warp; i < splits; i += kStatThreads / 32) {
            const int64_t at = (int64_t)i * n_lags + lag;
            if constexpr (WIDE)
                s.add(partial[at], low[at]);
            else
                s.add(partial[at]);
        }
    part_h[warp][lane] = s.high;
    part_l[warp][lane] = s.low;
    __syncthreads();
    if (warp != 0 || lag >= n_lags) return;
    for (int w = 1; w < kStatThreads / 32; ++w) s.add(part_h[w][lane], part_l[w][lane]);
    const double x = scalbn(scalbn(s.value(), -k), -k);
    const double v = x / ((double)n * (double)(len - lag)) / var;
    c[lag] = v;
    if (v <= 0.0) atomicMin(first, lag);
}

// events of level j in clone c: up-crossings to >= a, merged with an earlier
// one when the series was >= a within the last `gap` steps.  So step t >= 1 is
// an event if the series is >= a there and no step in the max(gap, 1) before it
// is.  A block per (clone, level), a warp per segment of the series, 32 steps a
// time by ballots (one thread per series took 1108 us, 64 x 6500); the first
// step >= a of each segment is judged against the segments before it at the end.
constexpr int kUpWarps = 8;

__global__ void __launch_bounds__(32 * kUpWarps) upcross_kernel(const double* drag, int32_t max_steps, int32_t t0,
                                                                int32_t len, const double* levels, int32_t gap,
                                                                unsigned long long* ev)
{
    __shared__ int count[kUpWarps], first[kUpWarps], last[kUpWarps];
    const int warp = threadIdx.x >> 5, lane = threadIdx.x & 31, quiet = max(gap, 1);
    const double a = levels[blockIdx.y];
    const double* row = drag + (int64_t)blockIdx.x * max_steps + t0;
    const int seg = ((len + kUpWarps - 1) / kUpWarps + 31) & ~31, b = min(warp * seg, len), e = min(b + seg, len);
    int n_ev = 0, head = -1, before = -1;  // before: the last step >= a so far
    for (int t = b; t < e; t += 32) {
        const bool up = t + lane < e && row[t + lane] >= a;
        const uint32_t m = __ballot_sync(0xffffffffu, up);
        if (m == 0u) continue;
        if (head < 0) head = t + __ffs(m) - 1;
        const uint32_t lower = m & ((1u << lane) - 1u);
        const int prev = lower ? t + 31 - __clz(lower) : before;
        n_ev += __popc(__ballot_sync(0xffffffffu, up && prev >= 0 && t + lane - prev > quiet));
        before = t + 31 - __clz(m);
    }
    if (lane == 0) {
        count[warp] = n_ev;
        first[warp] = head;
        last[warp] = before;
    }
    __syncthreads();
    if (threadIdx.x == 0) {
        unsigned long long total = 0;
        int prev = -1;
        for (int w = 0; w < kUpWarps; ++w) {
            if (first[w] < 0) continue;
            total += count[w] + (first[w] > 0 && (prev < 0 || first[w] - prev > quiet) ? 1 : 0);
            prev = last[w];
        }
        if (total) atomicAdd(ev + blockIdx.y, total);
    }
}

// A workspace of at least `bytes` for one call: the ensemble's own, grown on
// demand and kept until the ensemble is destroyed (used in its stream's order).
// A call that is being captured takes an allocation of the captured work itself
// instead, released behind it on every way out: the ensemble's own may have been
// replaced by a larger one when the captured work is replayed.
struct Workspace {
    char* p = nullptr;
    cudaStream_t captured = nullptr;
    bool temporary = false;
    Workspace() = default;
    Workspace(const Workspace&) = delete;
    Workspace& operator=(const Workspace&) = delete;
    ~Workspace()
    {
        if (temporary) cudaFreeAsync(p, captured);
    }
};

int stat_workspace(lbm_ensemble* e, size_t bytes, Workspace* ws)
{
    cudaStreamCaptureStatus capturing = cudaStreamCaptureStatusNone;
    LBM_CUDA(cudaStreamIsCapturing(e->stream, &capturing));
    if (capturing != cudaStreamCaptureStatusNone) {
        LBM_CUDA(cudaMallocAsync((void**)&ws->p, bytes, e->stream));
        ws->captured = e->stream;
        ws->temporary = true;
        return LBM_OK;
    }
    if (e->stat_bytes < bytes) {
        LBM_CUDA(cudaStreamSynchronize(e->stream));
        if (e->stat_ws) cudaFree(e->stat_ws);
        e->stat_ws = nullptr;
        e->stat_bytes = 0;
        LBM_CUDA(cudaMalloc(&e->stat_ws, bytes));
        e->stat_bytes = bytes;
    }
    ws->p = static_cast<char*>(e->stat_ws);
    return LBM_OK;
}

int check_window(lbm_ensemble* e, int32_t t0, int32_t t1)
{
    if (t0 < 0 || t1 <= t0 || t1 > e->cfg.max_steps) return fail(LBM_ERR_ARG, "drag statistics: need 0 <= t0 < t1 <= max_steps");
    for (int i = 0; i < e->n; ++i)
        if (e->t_host[i] < t1) return fail(LBM_ERR_STATE, "drag statistics: a clone has not reached t1");
    return LBM_OK;
}

}  // namespace
}  // namespace lbm

using namespace lbm;

extern "C" {

int lbm_drag_autocorrelation(lbm_ensemble* e, int32_t t0, int32_t t1, int32_t max_lag, double* c_dev, int32_t* tau_c)
{
    if (!e || !c_dev) return fail(LBM_ERR_ARG, "lbm_drag_autocorrelation: null argument");
    if (int rc = check_window(e, t0, t1)) return rc;
    if (max_lag < 0 || max_lag >= t1 - t0) return fail(LBM_ERR_ARG, "lbm_drag_autocorrelation: need 0 <= max_lag < t1 - t0");
    // workspace: moments of each clone, the limbs of the fluctuations (rows padded
    // so that a task's loads stay in its row), exact partial sums per split
    const int32_t len = t1 - t0, n = e->n, lags = max_lag + 1, pitch = (len + kCorrTime - 1) / kCorrTime * kCorrTime;
    const int lag_tiles = (lags + kCorrLags - 1) / kCorrLags;
    const int64_t tasks = (int64_t)n * (pitch / kCorrTime);
    if (tasks > INT32_MAX) return fail(LBM_ERR_ARG, "lbm_drag_autocorrelation: series too long");
    const int splits = (int)std::min<int64_t>(tasks, std::max(1, 152 * 12 / lag_tiles));
    const size_t limb_bytes = sizeof(int32_t) * (size_t)n * pitch, stat_bytes = (sizeof(double) * 3 * n + 15) / 16 * 16;
    const size_t sums = (size_t)splits * lags;
    const bool wide = (tasks + splits - 1) / splits > kCorrTasks;
    Workspace ws;
    if (int rc = stat_workspace(e, 16 + sizeof(__int128) * sums + (wide ? sizeof(long long) * sums : 0) + stat_bytes +
                                       2 * limb_bytes, &ws)) return rc;
    int32_t* first = reinterpret_cast<int32_t*>(ws.p);
    __int128* partial = reinterpret_cast<__int128*>(ws.p + 16);
    double* stat = reinterpret_cast<double*>(partial + sums);
    unsigned long long* low = reinterpret_cast<unsigned long long*>(ws.p + 16 + sizeof(__int128) * sums + stat_bytes +
                                                                    2 * limb_bytes);
    int32_t* hi = reinterpret_cast<int32_t*>(reinterpret_cast<char*>(stat) + stat_bytes);
    int32_t* lo = hi + (size_t)n * pitch;
    LBM_CUDA(cudaMemsetAsync(first, 0x7f, sizeof(int32_t), e->stream));
    drag_sum_kernel<<<n, kStatThreads, 0, e->stream>>>(e->drag, e->cfg.max_steps, t0, len, stat);
    drag_square_kernel<<<n, kStatThreads, 0, e->stream>>>(e->drag, e->cfg.max_steps, n, t0, len, stat);
    drag_limbs_kernel<<<dim3((pitch + kStatThreads - 1) / kStatThreads, n), kStatThreads, 0, e->stream>>>(
        e->drag, e->cfg.max_steps, n, t0, len, stat, pitch, hi, lo);
    auto correlate = [&](auto w) {
        constexpr bool WIDE = decltype(w)::value;
        autocorr_kernel<WIDE><<<dim3(lag_tiles, splits), kCorrThreads, 0, e->stream>>>(hi, lo, n, len, pitch, lags,
                                                                                     partial, low);
        autocorr_final_kernel<WIDE><<<(lags + 31) / 32, kStatThreads, 0, e->stream>>>(partial, low, splits, lags, stat,
                                                                                   n, len, c_dev, first);
    };
    if (wide)
        correlate(std::true_type{});
    else
        correlate(std::false_type{});
    LBM_CUDA(cudaGetLastError());
    count_launches(5);
    if (tau_c) {
        LBM_CUDA(cudaMemcpyAsync(tau_c, first, sizeof(int32_t), cudaMemcpyDeviceToHost, e->stream));
        LBM_CUDA(cudaStreamSynchronize(e->stream));
        if (*tau_c > max_lag) *tau_c = -1;
    }
    return LBM_OK;
}

int lbm_drag_return_times(lbm_ensemble* e, int32_t t0, int32_t t1, int32_t n_levels, const double* levels_dev,
                          int32_t gap, int64_t* events, double* r)
{
    if (!e || !levels_dev || !events || !r) return fail(LBM_ERR_ARG, "lbm_drag_return_times: null argument");
    if (int rc = check_window(e, t0, t1)) return rc;
    if (n_levels < 1 || n_levels > 4096 || gap < 0) return fail(LBM_ERR_ARG, "lbm_drag_return_times: levels or gap");
    Workspace ws;
    if (int rc = stat_workspace(e, sizeof(unsigned long long) * n_levels, &ws)) return rc;
    auto* ev = reinterpret_cast<unsigned long long*>(ws.p);
    LBM_CUDA(cudaMemsetAsync(ev, 0, sizeof(unsigned long long) * n_levels, e->stream));
    upcross_kernel<<<dim3(e->n, n_levels), 32 * kUpWarps, 0, e->stream>>>(e->drag, e->cfg.max_steps, t0, t1 - t0,
                                                                          levels_dev, gap, ev);
    LBM_CUDA(cudaGetLastError());
    count_launches(1);
    LBM_CUDA(cudaMemcpyAsync(events, ev, sizeof(int64_t) * n_levels, cudaMemcpyDeviceToHost, e->stream));
    LBM_CUDA(cudaStreamSynchronize(e->stream));
    const double observed = (double)e->n * (double)(t1 - t0);
    for (int j = 0; j < n_levels; ++j) {
        r[j] = events[j] > 0 ? observed / (double)events[j] : std::numeric_limits<double>::infinity();
    }
    return LBM_OK;
}

}  // extern "C"
