// Observables of the square, recorded after every step when enabled (Sec. 2.1
// and Sec. 3.2): the pressures integrated over its upstream face (forebody)
// and downstream face (base), whose difference approximates the drag (eq.
// drag_approx), and the mean wall shear d u_x / d y along its top and bottom
// faces (eq. avg_shear_def).  On the lattice, from the post-collision state
// of the step:
//   p_fb   = cs2 * sum over rows [oy0, oy1) of rho(ox0 - 1, y),
//   p_base = cs2 * sum over rows [oy0, oy1) of rho(ox1, y),
//   gamma_top    = mean over x in [ox0, ox1) of (9 u(x, oy1) - u(x, oy1 + 1)) / 3,
//   gamma_bottom = mean over x in [ox0, ox1) of -(9 u(x, oy0 - 1) - u(x, oy0 - 2)) / 3,
// the one-sided second-order slope at the halfway wall from the fluid rows at
// distances 1/2 and 3/2, with rho u = sum c f - F/2 (the post-collision
// momentum carries the step's whole force).  FP64 sums in a fixed order.
#include <cmath>

#include "internal.h"
#include "lbm_device.cuh"

namespace lbm {
namespace {

constexpr int kObsThreads = 128;

// sum of v[0 .. count) for the four quantities, one warp each: strided partial
// sums over kObsThreads, then a tree over them, in the order of a block-wide
// tree (the lanes hold entries l, l + 32, l + 64, l + 96 of it)
template <typename F>
__device__ double obs_warp_sum(int count, F&& v)
{
    double a[kObsThreads / 32];
#pragma unroll
    for (int k = 0; k < kObsThreads / 32; ++k) {
        a[k] = 0.0;
        for (int i = (threadIdx.x & 31) + 32 * k; i < count; i += kObsThreads) a[k] += v(i);
    }
    double s = (a[0] + a[2]) + (a[1] + a[3]);
#pragma unroll
    for (int off = 16; off > 0; off >>= 1) s += __shfl_down_sync(0xffffffffu, s, off);
    return s;
}

// density and velocity of node (x, y) of a post-collision state
template <int S>
__device__ void node_macro(const typename Codec<S>::T* st, int64_t plane, int32_t pitch, int x, int y, float inv_scale,
                           double hgx, double& rho, double& ux)
{
    const typename Codec<S>::T* cell = st + (int64_t)y * pitch + x;
    double drho = 0.0, jx = 0.0;
#pragma unroll
    for (int q = 0; q < 9; ++q) {
        const double g = (double)Codec<S>::dec(cell[q * plane], wf(q), inv_scale);
        drho += g;
        jx += cx(q) * g;
    }
    rho = 1.0 + drho;
    ux = (jx - hgx) / rho;
}

// One block per clone.  Latency bounds it: 96 nodes of a 16 x 16 square, FP64
// arithmetic at two operations a clock and SM.  With the nodes spread over the
// threads and one warp per sum it takes a fraction of the 16 us of a block that
// gave each of 16 threads six nodes in turn.
template <int S>
__global__ void __launch_bounds__(kObsThreads)
observables_kernel(const void* buf0, const void* buf1, const int32_t* parity, const int32_t* list, int32_t step,
                   int64_t clone_stride, int64_t plane, int32_t pitch, int32_t ox0, int32_t ox1, int32_t oy0,
                   int32_t oy1, double hgx, float inv_scale, const int32_t* t, double* obs, int32_t max_steps, bool staged)
{
    using T = typename Codec<S>::T;
    // the nodes the observables need, one per thread: the columns before and
    // after the square (densities), then four rows of its width (velocities):
    // above it at distances 1/2 and 3/2, below it at 1/2 and 3/2
    extern __shared__ double node[];
    const int c = list[blockIdx.x];
    const int cur = parity[c] ^ (step & 1);
    const T* st = static_cast<const T*>(cur ? buf0 : buf1) + (int64_t)c * clone_stride;  // this step's state
    constexpr double kCs2 = 1.0 / 3.0;
    const int h = oy1 - oy0, w = ox1 - ox0;
    auto value = [&](int i) {
        double rho, ux;
        if (i < 2 * h) {
            node_macro<S>(st, plane, pitch, i < h ? ox0 - 1 : ox1, oy0 + (i < h ? i : i - h), inv_scale, hgx, rho, ux);
            return rho;
        }
        const int k = (i - 2 * h) / w, x = ox0 + (i - 2 * h - k * w);
        const int y = k == 0 ? oy1 : (k == 1 ? oy1 + 1 : (k == 2 ? oy0 - 1 : oy0 - 2));
        node_macro<S>(st, plane, pitch, x, y, inv_scale, hgx, rho, ux);
        return ux;
    };
    if (staged)
        for (int i = threadIdx.x; i < 2 * h + 4 * w; i += kObsThreads) node[i] = value(i);
    __syncthreads();
    auto at = [&](int i) { return staged ? node[i] : value(i); };
    auto u = [&](int i) { return at(2 * h + i); };
    const int warp = threadIdx.x >> 5;
    double v;
    if (warp < 2)
        v = obs_warp_sum(h, [&](int i) { return kCs2 * at(warp * h + i); });
    else if (warp == 2)
        v = obs_warp_sum(w, [&](int i) { return (9.0 * u(i) - u(w + i)) / 3.0; });
    else
        v = obs_warp_sum(w, [&](int i) { return -((9.0 * u(2 * w + i) - u(3 * w + i)) / 3.0); });
    if ((threadIdx.x & 31) == 0) obs[((int64_t)c * max_steps + t[c] + step) * 4 + warp] = warp < 2 ? v : v / w;
}

}  // namespace

int observables_launch(lbm_ensemble* e, const int32_t* list_dev, int32_t n_list, int32_t step, cudaStream_t s)
{
    const lbm_config& c = e->cfg;
    const int ox0 = c.obs_x0, ox1 = c.obs_x0 + c.obs_w, oy0 = c.obs_y0, oy1 = c.obs_y0 + c.obs_h;
    const double hgx = 0.5 * c.gx;
    // a square whose nodes do not fit 48 KB is evaluated without staging them
    const size_t nodes = sizeof(double) * (2 * (size_t)c.obs_h + 4 * (size_t)c.obs_w);
    const bool staged = nodes <= 48 * 1024;
    const size_t smem = staged ? nodes : 0;
    switch (c.storage) {
    case kFP32:
        observables_kernel<kFP32><<<n_list, kObsThreads, smem, s>>>(e->buf[0], e->buf[1], e->parity_dev, list_dev, step,
                                                                 e->clone_stride, e->plane, e->pitch, ox0, ox1, oy0,
                                                                 oy1, hgx, e->inv_scale, e->t_dev, e->obs,
                                                                 c.max_steps, staged);
        break;
    case kFP16:
        observables_kernel<kFP16><<<n_list, kObsThreads, smem, s>>>(e->buf[0], e->buf[1], e->parity_dev, list_dev, step,
                                                                 e->clone_stride, e->plane, e->pitch, ox0, ox1, oy0,
                                                                 oy1, hgx, e->inv_scale, e->t_dev, e->obs,
                                                                 c.max_steps, staged);
        break;
    default:
        observables_kernel<kBF16><<<n_list, kObsThreads, smem, s>>>(e->buf[0], e->buf[1], e->parity_dev, list_dev, step,
                                                                 e->clone_stride, e->plane, e->pitch, ox0, ox1, oy0,
                                                                 oy1, hgx, e->inv_scale, e->t_dev, e->obs,
                                                                 c.max_steps, staged);
    }
    return cudaGetLastError() == cudaSuccess ? LBM_OK : LBM_ERR_CUDA;
}

}  // namespace lbm

using namespace lbm;

extern "C" {

int lbm_ensemble_set_observables(lbm_ensemble* e, int32_t enable)
{
    if (!e) return fail(LBM_ERR_ARG, "null ensemble");
    const lbm_config& c = e->cfg;
    if (enable) {
        if (c.obs_w <= 0 || c.obs_x0 < 1 || c.obs_x0 + c.obs_w > c.nx - 1 || c.obs_y0 < 2 ||
            c.obs_y0 + c.obs_h > c.ny - 2)
            return fail(LBM_ERR_ARG, "observables need a square with two fluid rows above and below it and a "
                                     "fluid column on either side");
        if (!e->obs) {
            const size_t bytes = sizeof(double) * 4 * (size_t)e->n * c.max_steps;
            LBM_CUDA(cudaMalloc((void**)&e->obs, bytes));
            LBM_CUDA(cudaMemsetAsync(e->obs, 0, bytes, e->stream));
        }
    }
    if ((enable != 0) != e->observe) {  // the captured step chunks change
        for (auto& g : e->graphs) cudaGraphExecDestroy(g.exec);
        e->graphs.clear();
    }
    e->observe = enable != 0;
    return LBM_OK;
}

int lbm_ensemble_observables(lbm_ensemble* e, int32_t t0, int32_t t1, double* dst, int32_t dst_on_device)
{
    if (!e || !dst) return fail(LBM_ERR_ARG, "null argument");
    if (!e->obs) return fail(LBM_ERR_STATE, "observables were never enabled");
    if (t0 < 0 || t1 < t0 || t1 > e->cfg.max_steps) return fail(LBM_ERR_ARG, "need 0 <= t0 <= t1 <= max_steps");
    const size_t row = sizeof(double) * 4 * (size_t)(t1 - t0);
    if (row == 0) return LBM_OK;
    const cudaMemcpyKind kind = dst_on_device ? cudaMemcpyDeviceToDevice : cudaMemcpyDeviceToHost;
    LBM_CUDA(cudaMemcpy2DAsync(dst, row, e->obs + (size_t)t0 * 4, sizeof(double) * 4 * (size_t)e->cfg.max_steps, row,
                               e->n, kind, e->stream));
    if (!dst_on_device) LBM_CUDA(cudaStreamSynchronize(e->stream));
    return LBM_OK;
}

}  // extern "C"
