// Kernels of the adjoint gradient (no counterpart in the paper, which
// differentiates through its TensorFlow backends only, Sec. 2.3):
//   * dot_partial_kernel: <phi|lambda> per member (the energy), FP64 across runs;
//   * grad_reduce_kernel: per-tile gradient partials -> dE/dtheta, FP64, fixed order.
// The costate seed lambda = H phi is kernels_hpsi.cu; the reverse sweep itself
// runs in the tiled pass kernel (TOP_GRAD ops).
#include <algorithm>
#include <cstring>

#include "adjoint.h"
#include "device.cuh"
#include "prof.h"

namespace qsim {

// ------------------------------------------------------------------ <a|b> per member
__device__ __forceinline__ double2 block_sum2_adj(double a, double b) {
    __shared__ double2 sh[32];
    for (int o = 16; o > 0; o >>= 1) {
        a += __shfl_down_sync(0xffffffffu, a, o);
        b += __shfl_down_sync(0xffffffffu, b, o);
    }
    const int lane = threadIdx.x & 31, warp = threadIdx.x >> 5;
    if (lane == 0) sh[warp] = make_double2(a, b);
    __syncthreads();
    double2 r = make_double2(0.0, 0.0);
    if (warp == 0) {
        const int nw = blockDim.x >> 5;
        r = lane < nw ? sh[lane] : make_double2(0.0, 0.0);
        for (int o = 16; o > 0; o >>= 1) {
            r.x += __shfl_down_sync(0xffffffffu, r.x, o);
            r.y += __shfl_down_sync(0xffffffffu, r.y, o);
        }
    }
    __syncthreads();
    return r;
}

template <typename R>
__global__ void __launch_bounds__(256) dot_partial_kernel(const V<R> *__restrict__ a, const V<R> *__restrict__ b,
                                                          int n, int ms, double2 *__restrict__ part) {
    const uint64_t per = 1ull << n;
    const V<R> *pa = a + ((uint64_t)blockIdx.y << ms);
    const V<R> *pb = b + ((uint64_t)blockIdx.y << ms);
    const uint64_t stride = (uint64_t)gridDim.x * blockDim.x;
    double sr = 0.0, si = 0.0;
    uint64_t i = (uint64_t)blockIdx.x * blockDim.x + threadIdx.x;
    while (i < per) {
        R rr = 0, ri = 0;
        for (int c = 0; c < 16 && i < per; ++c, i += stride) {
            const V<R> x = pa[i], y = pb[i];
            rr = fma(x.x, y.x, fma(x.y, y.y, rr));   // Re conj(x) y
            ri = fma(x.x, y.y, fma(-x.y, y.x, ri));  // Im conj(x) y
        }
        sr += (double)rr;
        si += (double)ri;
    }
    const double2 r = block_sum2_adj(sr, si);
    if (threadIdx.x == 0) part[(uint64_t)blockIdx.y * gridDim.x + blockIdx.x] = r;
}

__global__ void dot_finalize_kernel(const double2 *__restrict__ part, int per_member, double *__restrict__ out) {
    const int b = blockIdx.x;
    double x = 0.0, y = 0.0;
    for (int i = threadIdx.x; i < per_member; i += blockDim.x) {
        x += part[(uint64_t)b * per_member + i].x;
        y += part[(uint64_t)b * per_member + i].y;
    }
    const double2 r = block_sum2_adj(x, y);
    if (threadIdx.x == 0) {
        out[2 * b] = r.x;
        out[2 * b + 1] = r.y;
    }
}

qs_status k_dot(const StateView &a, const StateView &b, double *scratch, size_t scratch_doubles, double *out,
                cudaStream_t st) {
    int dev = 0, sms = 148;
    cudaGetDevice(&dev);
    cudaDeviceGetAttribute(&sms, cudaDevAttrMultiProcessorCount, dev);
    const uint64_t per = 1ull << a.n;
    int P = (int)std::min<uint64_t>(std::max<uint64_t>(1, per / (256 * 16)),
                                    std::max<uint64_t>(1, (uint64_t)sms * 8 / a.batch));
    P = (int)std::min<size_t>((size_t)P, std::max<size_t>(1, scratch_doubles / (2 * (size_t)a.batch)));
    ProfScope _ps(st, KC_ADJOINT, 2.0 * (double)((uint64_t)a.batch << a.n) * (a.dtype == QS_C64 ? 8 : 16),
                  8.0 * (double)((uint64_t)a.batch << a.n));
    dim3 grid(P, a.batch);
    if (a.dtype == QS_C64)
        dot_partial_kernel<float><<<grid, 256, 0, st>>>((const float2 *)a.data, (const float2 *)b.data, a.n, a.ms,
                                                        (double2 *)scratch);
    else
        dot_partial_kernel<double><<<grid, 256, 0, st>>>((const double2 *)a.data, (const double2 *)b.data, a.n,
                                                         a.ms, (double2 *)scratch);
    QS_CUDA_TRY(cudaGetLastError());
    dot_finalize_kernel<<<a.batch, 256, 0, st>>>((const double2 *)scratch, P, out);
    QS_CUDA_TRY(cudaGetLastError());
    return QS_OK;
}

// ------------------------------------------------------------------ gradient reduction
// grad[b * n_params + p] = sum over the gradient slots s of parameter p of
// coef[s] * sum over member b's tiles of part[s * total_tiles + tile], in a fixed
// order (slot list order, then a block reduction over tiles).
__global__ void __launch_bounds__(256) grad_reduce_kernel(const double *__restrict__ part,
                                                          const __grid_constant__ GradReduceP p,
                                                          double *__restrict__ grad) {
    const int pi = blockIdx.x, b = blockIdx.y;
    double total = 0.0;
    for (int k = p.beg[pi]; k < p.beg[pi + 1]; ++k) {
        const int s = p.slot[k];
        const double *row = part + (uint64_t)s * p.total_tiles + (uint64_t)b * p.tiles_per_member;
        double acc = 0.0;
        for (uint64_t t = threadIdx.x; t < p.tiles_per_member; t += blockDim.x) acc += row[t];
        const double2 r = block_sum2_adj(acc, 0.0);
        total += p.coef[k] * r.x;   // thread 0 holds the block sum
    }
    if (threadIdx.x == 0) grad[(uint64_t)b * p.n_params + p.param0 + pi] = total;
}

// The same with a warp per row: up to kWarpTiles tiles per member a CTA per row
// leaves most of its threads without a tile (n = 18, 64 members, 180 rows of 64
// tiles: 49 us; energy and gradient 2.98 -> 2.95 ms).
constexpr uint64_t kWarpTiles = 256;

__global__ void __launch_bounds__(256) grad_reduce_warp_kernel(const double *__restrict__ part,
                                                               const __grid_constant__ GradReduceP p, int rows,
                                                               double *__restrict__ grad) {
    const int pi = blockIdx.x * 8 + (threadIdx.x >> 5), b = blockIdx.y, lane = threadIdx.x & 31;
    if (pi >= rows) return;
    double total = 0.0;
    for (int k = p.beg[pi]; k < p.beg[pi + 1]; ++k) {
        const double *row = part + (uint64_t)p.slot[k] * p.total_tiles + (uint64_t)b * p.tiles_per_member;
        double acc = 0.0;
        for (uint64_t t = lane; t < p.tiles_per_member; t += 32) acc += row[t];
        for (int o = 16; o > 0; o >>= 1) acc += __shfl_down_sync(0xffffffffu, acc, o);
        total += p.coef[k] * acc;
    }
    if (lane == 0) grad[(uint64_t)b * p.n_params + p.param0 + pi] = total;
}

qs_status k_grad_reduce(const double *part, const GradReduceP &p, int n_param_rows, int batch, double *grad,
                        cudaStream_t st) {
    if (n_param_rows <= 0) return QS_OK;
    ProfScope _ps(st, KC_ADJOINT);
    if (p.tiles_per_member <= kWarpTiles)
        grad_reduce_warp_kernel<<<dim3((n_param_rows + 7) / 8, batch), 256, 0, st>>>(part, p, n_param_rows, grad);
    else
        grad_reduce_kernel<<<dim3(n_param_rows, batch), 256, 0, st>>>(part, p, grad);
    QS_CUDA_TRY(cudaGetLastError());
    return QS_OK;
}

}  // namespace qsim
