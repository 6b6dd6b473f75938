// adjoint.cu -- the adjoint of the masked log-joint of one data subset (an addition of this
// project; the paper samples with Gibbs only):
//   l(X, W, log a) = -(a/2) sum_{(n,d) in Omega} r_nd^2 + (|Omega|/2) log a
//                    - 1/2 sum_n (x_n - mu_n)^T L_n (x_n - mu_n) - 1/2 sum_d (w_d - mu_d)^T L_d (w_d - mu_d),
//   r_nd = y_nd - x_n^T w_d,
//   grad_x_n = a sum_{d in Omega_n} r_nd w_d - L_n (x_n - mu_n)   (and symmetrically for w_d),
//   dl/dlog a = |Omega|/2 - (a/2) sum r^2,
// where (mu_n, L_n) is the row's prior in the subset (the subset's hyperparameters, or the row's
// propagated Gaussian); terms constant in X, W and a are dropped from the value.
//
// FP32 arithmetic on FP32 factors, FP64 scalar sums.  Pass 1 (per side): one warp per work
// item (at most 1024 observations of one row).  K <= 16: lanes over observations, each lane
// gathers its partner row twice (dot product, then accumulation) and a butterfly
// reduce-scatter writes the item's K gradient entries and its sum of r^2.  K > 16: groups of
// 4 (K <= 32) or 8 (K <= 64) lanes per observation, eight features per lane, so that a partner
// row is read once, as consecutive 16-byte pieces; the dot product is reduced within the group
// and the gradient partial across the groups at the end of the item.  Pass 2: one warp per four
// rows (lanes over features) sums the rows' item partials in item order and adds the prior term,
// with the block's shared prior precision staged once in shared memory as FP32; per-block
// FP64 sums of r^2 and of the prior quadratic forms.  Deterministic.
#include <algorithm>

#include "common.cuh"
#include "kernels.h"

namespace bmf {

int adjoint_kt(int K) { return K <= 4 ? 4 : K <= 8 ? 8 : K <= 12 ? 12 : K <= 16 ? 16 : K <= 32 ? 32 : 64; }
int adjoint_ld(int K) { return (adjoint_kt(K) + 1 + 31) / 32 * 32; }

template <int C, int N>
__device__ __forceinline__ void rs_stepf(float (&acc)[N], int lane, int o)
{
    const bool up = (lane & o) != 0;
#pragma unroll
    for (int i = 0; i < C / 2; ++i) {
        float lo = acc[i], hi = acc[i + C / 2];
        float send = up ? lo : hi;
        float keep = up ? hi : lo;
        acc[i] = keep + __shfl_xor_sync(0xffffffffu, send, o);
    }
}

// Pass 1.  Row `row` of the "self" factor (arena numbering) is local row row - self0 of the
// caller's array; partner index idx (arena numbering of the other factor) is local idx - other0.
template <int KT>
__global__ void __launch_bounds__(256) adjoint_items_kernel(AdjointParams a)
{
    constexpr int LD = (KT + 1 + 31) / 32 * 32;
    const int lane = threadIdx.x & 31;
    const int64_t warp = ((int64_t)blockIdx.x * blockDim.x + threadIdx.x) >> 5;
    const int64_t nw = ((int64_t)gridDim.x * blockDim.x) >> 5;
    const int K = a.K;
    for (int64_t it = warp; it < a.n_items; it += nw) {
        const GramItem m = a.items[it];
        float x[KT];
        const float4 *xs = reinterpret_cast<const float4 *>(a.self + (int64_t)(m.row - a.self0) * a.ld);
#pragma unroll
        for (int v = 0; v < KT / 4; ++v) {
            const float4 q = __ldg(xs + v);
            x[4 * v] = 4 * v < K ? q.x : 0.f;
            x[4 * v + 1] = 4 * v + 1 < K ? q.y : 0.f;
            x[4 * v + 2] = 4 * v + 2 < K ? q.z : 0.f;
            x[4 * v + 3] = 4 * v + 3 < K ? q.w : 0.f;
        }
        float acc[LD];
#pragma unroll
        for (int v = 0; v < LD; ++v) acc[v] = 0.f;
        for (int e = lane; e < m.count; e += 32) {
            const int64_t q = m.begin + e;
            const int c = __ldg(a.idx + q) - a.other0;
            const float y = __ldg(a.val + q);
            const float4 *ps = reinterpret_cast<const float4 *>(a.other + (int64_t)c * a.ld);
            float dot = 0.f;
#pragma unroll
            for (int v = 0; v < KT / 4; ++v) {
                const float4 p = __ldg(ps + v);
                dot = fmaf(x[4 * v], p.x, dot);
                dot = fmaf(x[4 * v + 1], p.y, dot);
                dot = fmaf(x[4 * v + 2], p.z, dot);
                dot = fmaf(x[4 * v + 3], p.w, dot);
            }
            const float r = y - dot;
#pragma unroll
            for (int v = 0; v < KT / 4; ++v) {
                const float4 p = __ldg(ps + v);
                acc[4 * v] = fmaf(r, p.x, acc[4 * v]);
                acc[4 * v + 1] = fmaf(r, p.y, acc[4 * v + 1]);
                acc[4 * v + 2] = fmaf(r, p.z, acc[4 * v + 2]);
                acc[4 * v + 3] = fmaf(r, p.w, acc[4 * v + 3]);
            }
            acc[KT] = fmaf(r, r, acc[KT]);
        }
        rs_stepf<LD, LD>(acc, lane, 16);
        rs_stepf<LD / 2, LD>(acc, lane, 8);
        rs_stepf<LD / 4, LD>(acc, lane, 4);
        rs_stepf<LD / 8, LD>(acc, lane, 2);
        rs_stepf<LD / 16, LD>(acc, lane, 1);
        constexpr int PER = LD / 32;
        float *dst = a.part + it * (int64_t)LD + lane * PER;
#pragma unroll
        for (int v = 0; v < PER; ++v) dst[v] = acc[v];
    }
}

// Pass 1 for K > 16 (KT = 32 or 64): F = 8 features per lane, G = KT / F lanes per
// observation, 32 / G observations per warp step and two steps in flight.  Lane li of a group
// owns the two 16-byte pieces li and li + G of its row, so that one load of a group covers
// consecutive bytes: at KT = 64 a load touches one 128-byte line per observation, two per row (four
// when each lane owned 32 consecutive bytes).  The partner rows come from L2: 11.25 million
// observations at K = 64 take 226 us a side, 12.7 TB/s (231 us before).  A piece whose first
// feature is past K is not loaded (rows are 16-byte aligned with a pitch that is a multiple of 4
// floats and at least K, so every piece that is loaded lies inside its row).
template <int KT>
__global__ void __launch_bounds__(256) adjoint_items_grouped_kernel(AdjointParams a)
{
    constexpr int F = 8, PC = F / 4, G = KT / F, NG = 32 / G, LD = (KT + 1 + 31) / 32 * 32;
    static_assert(G * NG == 32 && G * F == KT, "group shape");
    const int lane = threadIdx.x & 31, g = lane / G, li = lane % G;
    const int64_t warp = ((int64_t)blockIdx.x * blockDim.x + threadIdx.x) >> 5;
    const int64_t nw = ((int64_t)gridDim.x * blockDim.x) >> 5;
    const int K = a.K;
    const int f0 = 4 * li;                     // piece j: features f0 + 4 G j ..
    for (int64_t it = warp; it < a.n_items; it += nw) {
        const GramItem m = a.items[it];
        float x[F];
        const float *xs = a.self + (int64_t)(m.row - a.self0) * a.ld + f0;
#pragma unroll
        for (int j = 0; j < PC; ++j) {
            float4 q = make_float4(0.f, 0.f, 0.f, 0.f);
            if (f0 + 4 * G * j < K) q = __ldg(reinterpret_cast<const float4 *>(xs + 4 * G * j));
            x[4 * j] = q.x;
            x[4 * j + 1] = q.y;
            x[4 * j + 2] = q.z;
            x[4 * j + 3] = q.w;
        }
#pragma unroll
        for (int f = 0; f < F; ++f)
            if (f0 + 4 * G * (f / 4) + f % 4 >= K) x[f] = 0.f;   // padding of the caller's rows is not read as data
        float acc[F];
#pragma unroll
        for (int f = 0; f < F; ++f) acc[f] = 0.f;
        float r2 = 0.f;
        for (int e0 = 0; e0 < m.count; e0 += 2 * NG) {
            const int ea = e0 + g, eb = e0 + NG + g;
            const bool va = ea < m.count, vb = eb < m.count;
            float ya = 0.f, yb = 0.f, pa[F], pb[F];
            const float *ra_row = nullptr, *rb_row = nullptr;
            if (va) {
                const int64_t q = m.begin + ea;
                ya = __ldg(a.val + q);
                ra_row = a.other + (int64_t)(__ldg(a.idx + q) - a.other0) * a.ld + f0;
            }
            if (vb) {
                const int64_t q = m.begin + eb;
                yb = __ldg(a.val + q);
                rb_row = a.other + (int64_t)(__ldg(a.idx + q) - a.other0) * a.ld + f0;
            }
#pragma unroll
            for (int j = 0; j < PC; ++j) {
                float4 u = make_float4(0.f, 0.f, 0.f, 0.f), v = u;
                if (va && f0 + 4 * G * j < K) u = __ldg(reinterpret_cast<const float4 *>(ra_row + 4 * G * j));
                if (vb && f0 + 4 * G * j < K) v = __ldg(reinterpret_cast<const float4 *>(rb_row + 4 * G * j));
                pa[4 * j] = u.x;
                pa[4 * j + 1] = u.y;
                pa[4 * j + 2] = u.z;
                pa[4 * j + 3] = u.w;
                pb[4 * j] = v.x;
                pb[4 * j + 1] = v.y;
                pb[4 * j + 2] = v.z;
                pb[4 * j + 3] = v.w;
            }
            float da = 0.f, db = 0.f;
#pragma unroll
            for (int f = 0; f < F; ++f) {
                da = fmaf(x[f], pa[f], da);
                db = fmaf(x[f], pb[f], db);
            }
#pragma unroll
            for (int o = G / 2; o >= 1; o >>= 1) {
                da += __shfl_xor_sync(0xffffffffu, da, o);
                db += __shfl_xor_sync(0xffffffffu, db, o);
            }
            // past the end of the item y = 0 and p = 0, so r = 0 adds nothing
            const float ra = ya - da, rb = yb - db;
#pragma unroll
            for (int f = 0; f < F; ++f) acc[f] = fmaf(rb, pb[f], fmaf(ra, pa[f], acc[f]));
            r2 = fmaf(rb, rb, fmaf(ra, ra, r2));
        }
        // sum over the groups (every lane of a group holds the group's r^2)
#pragma unroll
        for (int o = G; o < 32; o <<= 1) {
#pragma unroll
            for (int f = 0; f < F; ++f) acc[f] += __shfl_xor_sync(0xffffffffu, acc[f], o);
            r2 += __shfl_xor_sync(0xffffffffu, r2, o);
        }
        if (g == 0) {
            float *dst = a.part + it * (int64_t)LD + f0;
#pragma unroll
            for (int j = 0; j < PC; ++j)
                *reinterpret_cast<float4 *>(dst + 4 * G * j) =
                    make_float4(acc[4 * j], acc[4 * j + 1], acc[4 * j + 2], acc[4 * j + 3]);
            if (li == 0) a.part[it * (int64_t)LD + KT] = r2;
        }
    }
}

// Pass 2: a warp on four rows at a time (blocks step through the rows), lanes over the features.
// The prior precision and Lambda mu of the hyperparameter slot of the first row are staged once per
// block as FP32 in shared memory, zero-padded to KT columns (all rows of one side of a subset share
// the slot): an entry of the precision is read once for four rows, whose k-th features are one
// 16-byte broadcast.  Rows with another slot, or with their own propagated prior, read and convert
// their priors from global memory.  100,000 rows at K = 64: 123 us with a row per warp and a
// staged prior per 128 rows, 54 us with this (100,000 and 25,000 rows: 107 us together).
constexpr int kAdjWarps = 8;
constexpr int kAdjTile = 4;

template <int KT>
__global__ void __launch_bounds__(32 * kAdjWarps) adjoint_rows_kernel(AdjointParams a)
{
    constexpr int KP = KT + 1;    // odd pitch: lanes reading one column hit distinct banks
    constexpr int NI = (KT + 31) / 32;
    __shared__ float Lf[KT * KP], bf[KT];
    __shared__ __align__(16) float xs[kAdjWarps][KT][kAdjTile];
    const int K = a.K, LD = a.ldp;
    const int warp = threadIdx.x >> 5, lane = threadIdx.x & 31;
    const int hb = a.row_hslot[a.self0];
    if (hb >= 0) {
        const double *hp = a.hyper + (int64_t)hb * hyper_slot_len(K);
#pragma unroll 8
        for (int q = threadIdx.x; q < KT * KT; q += 32 * kAdjWarps) {
            const int i = q / KT, k = q % KT;
            Lf[i * KP + k] = (i < K && k < K) ? (float)hp[K + (i >= k ? tri(i, k) : tri(k, i))] : 0.f;
        }
        for (int q = threadIdx.x; q < KT; q += blockDim.x) bf[q] = q < K ? (float)hp[K + ntri(K) + q] : 0.f;
    }
    __syncthreads();
    double r2 = 0.0, quad = 0.0;
    for (int64_t n = ((int64_t)blockIdx.x * kAdjWarps + warp) * kAdjTile; n < a.n_rows;
         n += (int64_t)gridDim.x * kAdjWarps * kAdjTile) {
        const int nr = (int)min((int64_t)kAdjTile, a.n_rows - n);
        bool shared = hb >= 0;
        int64_t ip[kAdjTile + 1];
#pragma unroll
        for (int q = 0; q <= kAdjTile; ++q) ip[q] = a.item_ptr[a.self0 + n + min(q, nr)];
        float xv[kAdjTile][NI];
#pragma unroll
        for (int q = 0; q < kAdjTile; ++q) {
            shared = shared && (q >= nr || a.row_hslot[a.self0 + n + q] == hb);
#pragma unroll
            for (int u = 0; u < NI; ++u) {
                const int k = lane + 32 * u;
                xv[q][u] = q < nr && k < K ? a.self[(n + q) * a.ld + k] : 0.f;
            }
        }
        // data term: the row's item partials in order; r^2 rides in column KT
        float s[kAdjTile][NI];
#pragma unroll
        for (int q = 0; q < kAdjTile; ++q) {
#pragma unroll
            for (int u = 0; u < NI; ++u) s[q][u] = 0.f;
            const float *pt = a.part + (ip[q] - a.item_base) * (int64_t)LD;
            if (ip[q] < ip[q + 1]) {
#pragma unroll
                for (int u = 0; u < NI; ++u)
                    if (lane + 32 * u < KT) s[q][u] = pt[lane + 32 * u];
                if (lane == 0 && a.count_r2) r2 += (double)pt[KT];
            }
            // a heavy row's further items, four loads in flight
            for (int64_t left = ip[q + 1] - ip[q] - 1; left > 0; left -= 4) {
                float v[4][NI], w[4];
#pragma unroll
                for (int t = 0; t < 4; ++t) {
                    const float *src = pt + (t < left ? t + 1 : 0) * (int64_t)LD;
#pragma unroll
                    for (int u = 0; u < NI; ++u) v[t][u] = lane + 32 * u < KT ? src[lane + 32 * u] : 0.f;
                    w[t] = lane == 0 && a.count_r2 ? src[KT] : 0.f;
                }
#pragma unroll
                for (int t = 0; t < 4; ++t)
                    if (t < left) {
#pragma unroll
                        for (int u = 0; u < NI; ++u) s[q][u] += v[t][u];
                        if (lane == 0 && a.count_r2) r2 += (double)w[t];
                    }
                pt += 4 * (int64_t)LD;
            }
        }
#pragma unroll
        for (int q = 0; q < kAdjTile; ++q)
#pragma unroll
            for (int u = 0; u < NI; ++u)
                if (lane + 32 * u < KT) xs[warp][lane + 32 * u][q] = xv[q][u];
        __syncwarp();
        float qlane[kAdjTile] = {0.f, 0.f, 0.f, 0.f};
#pragma unroll
        for (int u = 0; u < NI; ++u) {
            const int i = lane + 32 * u;
            // prior term L (x - mu) = L x - b, in FP32 like the data term
            float l0[kAdjTile] = {0.f, 0.f, 0.f, 0.f}, l1[kAdjTile] = {0.f, 0.f, 0.f, 0.f};
            if (shared && i < KT) {
#pragma unroll 16
                for (int k = 0; k < KT; k += 2) {
                    const float la = Lf[i * KP + k], lb = Lf[i * KP + k + 1];
                    const float4 v = *reinterpret_cast<const float4 *>(xs[warp][k]);
                    const float4 w = *reinterpret_cast<const float4 *>(xs[warp][k + 1]);
                    l0[0] = fmaf(la, v.x, l0[0]), l1[0] = fmaf(lb, w.x, l1[0]);
                    l0[1] = fmaf(la, v.y, l0[1]), l1[1] = fmaf(lb, w.y, l1[1]);
                    l0[2] = fmaf(la, v.z, l0[2]), l1[2] = fmaf(lb, w.z, l1[2]);
                    l0[3] = fmaf(la, v.w, l0[3]), l1[3] = fmaf(lb, w.w, l1[3]);
                }
            }
            if (i < K) {
#pragma unroll
                for (int q = 0; q < kAdjTile; ++q) {
                    if (q >= nr) break;
                    float lx = l0[q] + l1[q], b = bf[i];
                    if (!shared) {
                        const int64_t row = a.self0 + n + q;
                        const int h = a.row_hslot[row];
                        const double *hp = h >= 0 ? a.hyper + (int64_t)h * hyper_slot_len(K) : nullptr;
                        lx = 0.f;
                        for (int k = 0; k < K; ++k) {
                            const int e = i >= k ? tri(i, k) : tri(k, i);
                            const float l = (float)(hp ? hp[K + e] : a.prior_L[(int64_t)e * a.R + row]);
                            lx = fmaf(l, xs[warp][k][q], lx);
                        }
                        b = (float)(hp ? hp[K + ntri(K) + i] : a.prior_b[(int64_t)i * a.R + row]);
                    }
                    a.grad[(n + q) * a.ld + i] = (float)a.alpha * s[q][u] - (lx - b);
                    // (x - mu)^T L (x - mu) = x^T L x - 2 x^T b + mu^T b: the last term is constant
                    qlane[q] = fmaf(xv[q][u], lx - 2.f * b, qlane[q]);
                }
            }
        }
#pragma unroll
        for (int q = 0; q < kAdjTile; ++q) {
            if (q >= nr) break;
            for (int i = K + lane; i < a.ld; i += 32) a.grad[(n + q) * a.ld + i] = 0.f;
            float v = qlane[q];
#pragma unroll
            for (int o = 16; o >= 1; o >>= 1) v += __shfl_xor_sync(0xffffffffu, v, o);
            if (lane == 0) quad += (double)v;
        }
        __syncwarp();   // xs is rewritten for the next rows
    }
    __shared__ double red[2][kAdjWarps];
    if (lane == 0) {
        red[0][warp] = r2;
        red[1][warp] = quad;
    }
    __syncthreads();
    if (threadIdx.x == 0) {
        double s0 = 0.0, s1 = 0.0;
        for (int w = 0; w < kAdjWarps; ++w) {
            s0 += red[0][w];
            s1 += red[1][w];
        }
        a.block_sums[2 * blockIdx.x] = s0;
        a.block_sums[2 * blockIdx.x + 1] = s1;
    }
}

// Blocks of pass 2: a quarter of an SM each where a prior of 16 KB is staged per block, an eighth
// where it is small; no more than the rows fill.
int adjoint_row_blocks(int64_t n_rows, int kt, int sms)
{
    const int64_t most = (int64_t)(kt >= 32 ? 4 : 8) * sms;
    return (int)std::min<int64_t>((n_rows + kAdjWarps * kAdjTile - 1) / (kAdjWarps * kAdjTile), most);
}

// The two scalar sums of every block of both sides, in order within a fixed split and tree.
__global__ void __launch_bounds__(256) adjoint_sums_kernel(const double *sums, int n, double *out)
{
    __shared__ double red[2][256];
    double s0 = 0.0, s1 = 0.0;
    for (int b = threadIdx.x; b < n; b += 256) {
        s0 += sums[2 * b];
        s1 += sums[2 * b + 1];
    }
    red[0][threadIdx.x] = s0;
    red[1][threadIdx.x] = s1;
    __syncthreads();
    for (int o = 128; o > 0; o >>= 1) {
        if (threadIdx.x < o) {
            red[0][threadIdx.x] += red[0][threadIdx.x + o];
            red[1][threadIdx.x] += red[1][threadIdx.x + o];
        }
        __syncthreads();
    }
    if (threadIdx.x < 2) out[threadIdx.x] = red[threadIdx.x][0];
}

void launch_adjoint_sums(const double *sums, int n, double *out, cudaStream_t st)
{
    adjoint_sums_kernel<<<1, 256, 0, st>>>(sums, n, out);
}

template <int KT>
static void launch_items_t(const AdjointParams &a, int grid, cudaStream_t st)
{
    if constexpr (KT >= 32)
        adjoint_items_grouped_kernel<KT><<<grid, 256, 0, st>>>(a);
    else
        adjoint_items_kernel<KT><<<grid, 256, 0, st>>>(a);
}

void launch_adjoint(const AdjointParams &a, int grid, cudaStream_t st)
{
    if (a.n_items > 0) {
        switch (a.kt) {
        case 4: launch_items_t<4>(a, grid, st); break;
        case 8: launch_items_t<8>(a, grid, st); break;
        case 12: launch_items_t<12>(a, grid, st); break;
        case 16: launch_items_t<16>(a, grid, st); break;
        case 32: launch_items_t<32>(a, grid, st); break;
        default: launch_items_t<64>(a, grid, st); break;
        }
    }
    if (a.n_rows > 0) {
        const int blocks = a.row_blocks;
        switch (a.kt) {
        case 4: adjoint_rows_kernel<4><<<blocks, 32 * kAdjWarps, 0, st>>>(a); break;
        case 8: adjoint_rows_kernel<8><<<blocks, 32 * kAdjWarps, 0, st>>>(a); break;
        case 12: adjoint_rows_kernel<12><<<blocks, 32 * kAdjWarps, 0, st>>>(a); break;
        case 16: adjoint_rows_kernel<16><<<blocks, 32 * kAdjWarps, 0, st>>>(a); break;
        case 32: adjoint_rows_kernel<32><<<blocks, 32 * kAdjWarps, 0, st>>>(a); break;
        default: adjoint_rows_kernel<64><<<blocks, 32 * kAdjWarps, 0, st>>>(a); break;
        }
    }
}

// Langevin move on the FP32 factors X and W: out = theta + (eps/2) grad + sqrt(eps) xi (out may be
// theta itself; padding is kept, and copied where out is not theta).
__global__ void langevin_kernel(const float *X, const float *W, const float *gX, const float *gW, float *oX,
                                float *oW, const float *xi, int64_t n_x, int64_t n_w, int K, int ld, float eps)
{
    const int64_t q = (int64_t)blockIdx.x * blockDim.x + threadIdx.x;
    if (q >= (n_x + n_w) * ld) return;
    const int64_t r = q / ld;
    const int k = (int)(q % ld);
    const bool x = r < n_x;
    const int64_t o = x ? q : q - n_x * ld;
    const float *t = x ? X : W, *g = x ? gX : gW;
    float *d = x ? oX : oW;
    if (k < K)
        d[o] = t[o] + 0.5f * eps * g[o] + sqrtf(eps) * xi[r * K + k];
    else if (d != t)
        d[o] = t[o];
}

void launch_langevin(const float *X, const float *W, const float *gX, const float *gW, float *oX, float *oW,
                     const float *xi, int64_t n_x, int64_t n_w, int K, int ld, float eps, cudaStream_t st)
{
    const int64_t n = (n_x + n_w) * ld;
    if (n > 0)
        langevin_kernel<<<(int)((n + 255) / 256), 256, 0, st>>>(X, W, gX, gW, oX, oW, xi, n_x, n_w, K, ld, eps);
}

// FP32 copy of FP64 observation values (for contexts that gather in FP64).
__global__ void to_float_kernel(const double *in, float *out, int64_t n)
{
    const int64_t q = (int64_t)blockIdx.x * blockDim.x + threadIdx.x;
    if (q < n) out[q] = (float)in[q];
}

void launch_to_float(const double *in, float *out, int64_t n, cudaStream_t st)
{
    if (n > 0) to_float_kernel<<<(int)((n + 255) / 256), 256, 0, st>>>(in, out, n);
}

// Per-block FP64 sums of sum_k (a - b - coef g)^2 over rows x K (row pitch ld).
__global__ void __launch_bounds__(256) sqdiff_kernel(const float *a, const float *b, const float *g,
                                                     double coef, int64_t n_rows, int K,
                                                     int64_t ld, double *block_sums)
{
    double s = 0.0;
    const int64_t n = n_rows * K;
    for (int64_t q = (int64_t)blockIdx.x * blockDim.x + threadIdx.x; q < n;
         q += (int64_t)gridDim.x * blockDim.x) {
        const int64_t o = (q / K) * ld + q % K;
        const double d = (double)a[o] - (double)b[o] - coef * (double)g[o];
        s += d * d;
    }
    __shared__ double red[256];
    red[threadIdx.x] = s;
    __syncthreads();
    for (int o = 128; o > 0; o >>= 1) {
        if (threadIdx.x < o) red[threadIdx.x] += red[threadIdx.x + o];
        __syncthreads();
    }
    if (threadIdx.x == 0) block_sums[blockIdx.x] = red[0];
}

void launch_sqdiff(const float *a, const float *b, const float *g, double coef, int64_t n_rows,
                   int K, int64_t ld, double *block_sums, int blocks, cudaStream_t st)
{
    sqdiff_kernel<<<blocks, 256, 0, st>>>(a, b, g, coef, n_rows, K, ld, block_sums);
}

}  // namespace bmf
