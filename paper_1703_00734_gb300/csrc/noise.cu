// noise.cu -- the sampled noise precision (Section 2.1: one precision tau_d per column, or one
// per chain, with conjugate Gamma(a0, b0) priors, shape and rate):
//   tau_d | X, W ~ Gamma(a0 + n_d / 2, b0 + SSE_d / 2),  SSE_d = sum_{n in Omega_d} (y_nd -
//   x_n^T w_d)^2,  drawn as c / (2 b0 + SSE_d) from a chi-square variate c with 2 a0 + n_d
//   degrees of freedom (one precision: the subset's entries and summed SSE).
// The row-side Gram pass takes the per-column precisions through scaled copies: partner rows
// sqrt(tau_d) w_d and values sqrt(tau_d) y_nd, so that sum (sqrt(tau) w)(sqrt(tau) w)^T =
// sum tau w w^T and sum (sqrt(tau) y)(sqrt(tau) w) = sum tau y w.
#include <cuda_bf16.h>

#include "common.cuh"
#include "kernels.h"

namespace bmf {

// Squared residuals of one Gram work item (at most 1024 entries of one column) per warp: lanes
// over the item's entries, each lane reading its partner's FP64 state row; the column's own row
// is uniform over the warp.  A warp's FP64 instruction costs the same whatever its active lanes,
// so lanes over entries (K + 2 FP64 instructions per 32 entries) beats lanes over features with
// a shuffled sum, and splitting heavy columns over items bounds the longest serial chain at 32
// entries.  A thread per column, the earlier form, waits for the heaviest column: 20 sweeps of a
// 30,011 x 2,027 Zipf matrix with 900,000 entries at K = 24 (TF32 gathers, whole call) took
// 882 ms with it and take 28.5 ms with this.  The lane sums are added in a
// butterfly and a column's items in order: a fixed order.
template <typename VT, bool EVEN>
__global__ void __launch_bounds__(256) noise_sse_kernel(int K, const GramItem *items, int64_t n_items,
                                                        const int32_t *idx, const VT *val,
                                                        const double *X, const double *W, double *part)
{
    const int lane = threadIdx.x & 31;
    const int64_t nw = ((int64_t)gridDim.x * blockDim.x) >> 5;
    for (int64_t it = (int64_t)(threadIdx.x >> 5) * gridDim.x + blockIdx.x; it < n_items; it += nw) {
        const GramItem m = items[it];
        const double *w = W + (int64_t)m.row * K;
        double s = 0.0;
        for (int e = lane; e < m.count; e += 32) {
            const int64_t q = m.begin + e;
            const double *x = X + (int64_t)__ldg(idx + q) * K;
            double p0 = 0.0, p1 = 0.0;
            if constexpr (EVEN) {   // rows of an even K start on 16-byte boundaries
#pragma unroll 4
                for (int k = 0; k < K; k += 2) {
                    const double2 u = __ldg(reinterpret_cast<const double2 *>(x + k));
                    const double2 v = __ldg(reinterpret_cast<const double2 *>(w + k));
                    p0 = fma(u.x, v.x, p0);
                    p1 = fma(u.y, v.y, p1);
                }
            } else {
#pragma unroll 4
                for (int k = 0; k < K; ++k) p0 = fma(__ldg(x + k), __ldg(w + k), p0);
            }
            const double r = (double)__ldg(val + q) - (p0 + p1);
            s = fma(r, r, s);
        }
#pragma unroll
        for (int o = 16; o >= 1; o >>= 1) s += __shfl_xor_sync(0xffffffffu, s, o);
        if (lane == 0) part[it] = s;
    }
}

template <typename VT>
static void launch_sse_t(int K, const GramItem *items, int64_t n_items, const int32_t *idx,
                         const VT *val, const double *X, const double *W, double *part, int sms,
                         cudaStream_t st)
{
    const int grid = (int)(n_items < (int64_t)sms * 8 ? n_items : (int64_t)sms * 8);
    if (K % 2 == 0)
        noise_sse_kernel<VT, true><<<grid, 256, 0, st>>>(K, items, n_items, idx, val, X, W, part);
    else
        noise_sse_kernel<VT, false><<<grid, 256, 0, st>>>(K, items, n_items, idx, val, X, W, part);
}

void launch_noise_sse(int K, const GramItem *items, int64_t n_items, const int32_t *idx,
                      const void *val, int prec, const double *X, const double *W, double *part,
                      int sms, cudaStream_t st)
{
    if (n_items <= 0) return;
    if (prec == BMF_FP64)
        launch_sse_t(K, items, n_items, idx, static_cast<const double *>(val), X, W, part, sms, st);
    else
        launch_sse_t(K, items, n_items, idx, static_cast<const float *>(val), X, W, part, sms, st);
}

// Column mode (blocks over the rows of each subset): a row's items in order, then its
// precision.  Global mode (one block per subset): the subset's items in a fixed strided split and
// tree, then one precision to every row.
__global__ void __launch_bounds__(256) noise_tau_kernel(int mode, double b0, const NoiseBlock *blocks,
                                                        const double *draws, const double *part,
                                                        const int64_t *item_ptr, int64_t item0,
                                                        double *tau)
{
    const NoiseBlock b = blocks[blockIdx.x];
    if (mode == 2) {
        for (int64_t r = b.r0 + (int64_t)blockIdx.y * blockDim.x + threadIdx.x; r < b.r1;
             r += (int64_t)gridDim.y * blockDim.x) {
            double s = 0.0;
            for (int64_t it = item_ptr[r]; it < item_ptr[r + 1]; ++it) s += part[it - item0];
            tau[r] = draws[b.draw + (r - b.r0)] / (2.0 * b0 + s);
        }
        return;
    }
    __shared__ double red[256];
    double s = 0.0;
    for (int64_t it = item_ptr[b.r0] + threadIdx.x; it < item_ptr[b.r1]; it += blockDim.x)
        s += part[it - item0];
    red[threadIdx.x] = s;
    __syncthreads();
    for (int o = 128; o > 0; o >>= 1) {
        if (threadIdx.x < o) red[threadIdx.x] += red[threadIdx.x + o];
        __syncthreads();
    }
    const double t = draws[b.draw] / (2.0 * b0 + red[0]);
    for (int64_t r = b.r0 + threadIdx.x; r < b.r1; r += blockDim.x) tau[r] = t;
}

void launch_noise_tau(int mode, double b0, const NoiseBlock *blocks, int n_blocks,
                      const double *draws, const double *part, const int64_t *item_ptr,
                      int64_t item0, double *tau, cudaStream_t st)
{
    if (n_blocks <= 0) return;
    noise_tau_kernel<<<dim3(n_blocks, mode == 2 ? 32 : 1), 256, 0, st>>>(mode, b0, blocks, draws, part,
                                                                        item_ptr, item0, tau);
}

template <typename GT>
__device__ __forceinline__ GT to_g(double x);
template <>
__device__ __forceinline__ double to_g<double>(double x) { return x; }
template <>
__device__ __forceinline__ float to_g<float>(double x) { return (float)x; }
template <>
__device__ __forceinline__ __nv_bfloat16 to_g<__nv_bfloat16>(double x) { return __double2bfloat16(x); }

template <typename GT, typename VT>
__global__ void noise_scale_kernel(int K, int64_t r0, int64_t r1, const double *tau, const double *W,
                                   GT *Ws, int ldg, int64_t q0, int64_t q1, const int32_t *idx,
                                   const VT *val_orig, VT *val)
{
    const int64_t i = (int64_t)blockIdx.x * blockDim.x + threadIdx.x;
    const int64_t nrow = (r1 - r0) * ldg;
    if (i < nrow) {
        const int64_t r = r0 + i / ldg;
        const int k = (int)(i % ldg);
        Ws[r * ldg + k] = to_g<GT>(k < K ? sqrt(tau[r]) * W[r * K + k] : 0.0);
        return;
    }
    const int64_t q = q0 + (i - nrow);
    if (q < q1) val[q] = (VT)((double)val_orig[q] * sqrt(tau[idx[q]]));
}

void launch_noise_scale(int K, int prec, int64_t r0, int64_t r1, const double *tau,
                        const double *W, void *Ws, int ldg, int64_t q0, int64_t q1,
                        const int32_t *idx, const void *val_orig, void *val, cudaStream_t st)
{
    const int64_t n = (r1 - r0) * ldg + (q1 - q0);
    if (n <= 0) return;
    const int grid = (int)((n + 255) / 256);
    if (prec == BMF_FP64)
        noise_scale_kernel<double, double><<<grid, 256, 0, st>>>(
            K, r0, r1, tau, W, (double *)Ws, ldg, q0, q1, idx, (const double *)val_orig, (double *)val);
    else if (prec == BMF_FP32)
        noise_scale_kernel<float, float><<<grid, 256, 0, st>>>(
            K, r0, r1, tau, W, (float *)Ws, ldg, q0, q1, idx, (const float *)val_orig, (float *)val);
    else
        noise_scale_kernel<__nv_bfloat16, float><<<grid, 256, 0, st>>>(
            K, r0, r1, tau, W, (__nv_bfloat16 *)Ws, ldg, q0, q1, idx, (const float *)val_orig,
            (float *)val);
}

}  // namespace bmf
