// gram.cu -- the Gram-gather pass of the Gibbs sweep: for every arena row n (or a chunk of a
// long row), G_n = sum_{d in Omega_n} p_d p_d^T and r_n = sum_{d in Omega_n} y_nd p_d, where p_d
// are the gathered latent vectors of the observed partners (the row-side and column-side
// conditionals of BPMF, Eqs. 2-4; the MK^2 term of the cost model of Section 4.3).
//
// A warp task is one long work item (32 lanes) or several short rows (groups of 16 or 8 lanes,
// one row per group).  Lanes of a group stride over the row's observations and gather one
// partner row each with vector loads (the number of scattered load requests, not bytes, bounds
// a gather on this GPU), accumulating the packed-lower Gram entries and the right-hand side in
// registers; a butterfly
// reduce-scatter within the group then leaves each lane with a slice of the summed entries.
// Entries are split into parts of EP values when they do not fit in registers.  Rows longer than
// one item are finished by the warp that completes their last item.  Every sum has a fixed order:
// results are deterministic.
#include <cuda_bf16.h>

#include "common.cuh"
#include "kernels.h"

namespace bmf {

int padded_k(int K) { return K <= 1 ? 2 : (K + 1) / 2 * 2; }

// Gathered rows start on 16-byte boundaries (128-bit loads).
int gather_ld(int K, int prec)
{
    if (K > 16) return wide_kt(K);   // rows of 32, 48 or 64 elements (16-byte multiples)
    const int KT = padded_k(K);
    const int per16 = prec == BMF_FP64 ? 2 : (prec == BMF_BF16 ? 8 : 4);
    return (KT + per16 - 1) / per16 * per16;
}

// The latent dimension a kernel is compiled for: K itself in FP64, where the pass is bound by its
// FP64 instructions (K = 5: 20 sums, 27 padded to K = 6: 54,000 rows of 74 observations 358 -> 265
// us with the uneven reduce-scatter), K rounded up to an even number else.
__host__ __device__ constexpr int width_of(int K, bool fp64) { return fp64 ? K : (K <= 1 ? 2 : (K + 1) / 2 * 2); }

// Entries per part: FP32 registers hold all of a lane's accumulators (up to 160, in one part); FP64
// takes as few equal parts of at most 32 as hold them (K = 10: 22 each; 32 + 32 + 1 gathered every
// row a third time for one sum).
__host__ __device__ constexpr int parts_of(int KT, bool fp64) { return fp64 ? (gram_nv(KT) + 31) / 32 : 1; }
__host__ __device__ constexpr int ep_of(int KT, bool fp64)
{
    return fp64 ? (gram_nv(KT) + parts_of(KT, true) - 1) / parts_of(KT, true) : (gram_nv(KT) <= 96 ? 96 : 160);
}

int gram_width(int K, int prec) { return width_of(K, prec == BMF_FP64); }

int gram_parts(int K, int prec) { return parts_of(gram_width(K, prec), prec == BMF_FP64); }

int gram_part_ld(int K, int prec)
{
    return prec == BMF_FP64 ? (gram_nv(K) + 1) / 2 * 2 : ep_of(gram_width(K, prec), false);
}

// Lanes per row by its observation count: fewer lanes per row means more rows per warp and a
// shorter reduce-scatter per row; measured on this GPU (69,878 x 10,677 Zipf workload, K = 10)
// the X-side pass took 118 us with these thresholds against 140 us with (16, 48).
int gram_group(int64_t count) { return count <= 64 ? 8 : (count <= 256 ? 16 : 32); }

__device__ __forceinline__ float madd(float a, float b, float c) { return fmaf(a, b, c); }
__device__ __forceinline__ double madd(double a, double b, double c) { return fma(a, b, c); }

// ------------------------------------------------------------------------------------------
// Row gathers: the first BYTES bytes of a 16-byte aligned row with 128-bit loads (a tail of at
// most 8 bytes with one 64-bit load).  Measured on this GPU: 256-bit loads at a 32-byte row
// pitch were slower here than 128-bit loads at the tighter 16-byte pitch (fewer L1 hits on the
// frequently gathered rows).
// ------------------------------------------------------------------------------------------
template <int BYTES>
__device__ __forceinline__ void load_bits(const void *__restrict__ p, uint32_t (&u)[(BYTES + 3) / 4])
{
    constexpr int NW = (BYTES + 3) / 4;
    const uint4 *q = static_cast<const uint4 *>(p);
    constexpr int FULL = BYTES / 16, REM = BYTES - 16 * FULL;
    constexpr int N16 = FULL + (REM > 8 ? 1 : 0);
#pragma unroll
    for (int c = 0; c < N16; ++c) {
        const uint4 v = __ldg(q + c);
        const uint32_t w[4] = {v.x, v.y, v.z, v.w};
#pragma unroll
        for (int k = 0; k < 4; ++k)
            if (4 * c + k < NW) u[4 * c + k] = w[k];
    }
    if constexpr (REM > 0 && REM <= 8) {
        const uint2 v = __ldg(reinterpret_cast<const uint2 *>(q + FULL));
        u[4 * FULL] = v.x;
        if (4 * FULL + 1 < NW) u[4 * FULL + 1] = v.y;
    }
}

template <int K>
__device__ __forceinline__ void load_row(const float *__restrict__ p, float (&w)[K])
{
    uint32_t u[K];
    load_bits<4 * K>(p, u);
#pragma unroll
    for (int k = 0; k < K; ++k) w[k] = __uint_as_float(u[k]);
}
template <int K>
__device__ __forceinline__ void load_row(const double *__restrict__ p, double (&w)[K])
{
    uint32_t u[2 * K];
    load_bits<8 * K>(p, u);
#pragma unroll
    for (int k = 0; k < K; ++k) w[k] = __hiloint2double((int)u[2 * k + 1], (int)u[2 * k]);
}
template <int K>
__device__ __forceinline__ void load_row(const __nv_bfloat16 *__restrict__ p, float (&w)[K])
{
    uint32_t u[(K + 1) / 2];
    load_bits<2 * K>(p, u);
#pragma unroll
    for (int k = 0; k < K; ++k)
        w[k] = __uint_as_float(k & 1 ? u[k / 2] & 0xffff0000u : u[k / 2] << 16);
}

// ------------------------------------------------------------------------------------------
// Accumulation and the in-group reduce-scatter
// ------------------------------------------------------------------------------------------

// One butterfly step over C values: the lane half selected by bit `o` keeps the upper half of
// the values, the other the lower half; each adds its partner's copy.
template <int C, int N, typename AT>
__device__ __forceinline__ void rs_step(AT (&acc)[N], int lane, int o)
{
    const bool up = (lane & o) != 0;
#pragma unroll
    for (int i = 0; i < C / 2; ++i) {
        AT lo = acc[i], hi = acc[i + C / 2];
        AT send = up ? lo : hi;
        AT keep = up ? hi : lo;
        acc[i] = keep + __shfl_xor_sync(0xffffffffu, send, o);
    }
}

// Steps with offsets O, O/2, ..., 1 (a group of 2*O lanes); afterwards lane li of the group
// holds the entries [li * C0 / (2*O), (li + 1) * C0 / (2*O)) of the group's sum.
template <int C, int O, int N, typename AT>
__device__ __forceinline__ void rs_group(AT (&acc)[N], int lane)
{
    if constexpr (O >= 1) {
        rs_step<C, N, AT>(acc, lane, O);
        rs_group<C / 2, O / 2, N, AT>(acc, lane);
    }
}

// The same for a count that need not divide (FP64, where every addition counts): the lanes with
// bit O keep the upper values [H, C), the others the lower [0, H), H = ceil(C / 2); each adds its
// partner's copy.  Afterwards a lane holds scattered<C, O>() values of the group's sums from
// `base` on, those below `end`.
template <int C, int O>
__host__ __device__ constexpr int scattered()
{
    if constexpr (O >= 1)
        return scattered<(C + 1) / 2, O / 2>();
    else
        return C;
}
template <int C, int O, int N, typename AT>
__device__ __forceinline__ void rs_uneven(AT (&acc)[N], int lane, int &base, int &end)
{
    if constexpr (O >= 1) {
        constexpr int H = (C + 1) / 2;
        const bool up = (lane & O) != 0;
#pragma unroll
        for (int i = 0; i < H; ++i) {
            const AT lo = acc[i], hi = i + H < C ? acc[i + H < C ? i + H : 0] : AT(0);
            const AT send = up ? lo : hi;
            const AT keep = up ? hi : lo;
            acc[i] = keep + __shfl_xor_sync(0xffffffffu, send, O);
        }
        if (up)
            base += H;
        else
            end = min(end, base + H);
        rs_uneven<H, O / 2, N, AT>(acc, lane, base, end);
    }
}

// Gram entry E (packed lower (i, j), then right-hand side) for one observation.
template <int KT, int E, typename AT>
__device__ __forceinline__ void accum_entry(AT &acc, const AT (&w)[KT], AT y)
{
    constexpr int NT = ntri(KT);
    if constexpr (E < NT) {
        constexpr int i = [] {
            int r = 0;
            while ((r + 1) * (r + 2) / 2 <= E) ++r;
            return r;
        }();
        constexpr int j = E - i * (i + 1) / 2;
        acc = madd(w[i], w[j], acc);
    } else if constexpr (E < NT + KT) {
        acc = madd(y, w[E - NT], acc);
    }
}

template <int KT, int EP, int BASE, int I, typename AT>
__device__ __forceinline__ void accum_all(AT (&acc)[EP], const AT (&w)[KT], AT y)
{
    if constexpr (I < EP) {
        accum_entry<KT, BASE + I, AT>(acc[I], w, y);
        accum_all<KT, EP, BASE, I + 1, AT>(acc, w, y);
    }
}

// One warp task with groups of G lanes: group g handles item tk.item0 + g (g < tk.n).
template <int KT, typename GT, typename AT, int EP, int PART, int G>
__device__ __forceinline__ void gram_task(const GramParams &a, const GramTask &tk, int lane)
{
    const GT *__restrict__ P = static_cast<const GT *>(a.P);
    const AT *__restrict__ val = static_cast<const AT *>(a.val);
    AT *__restrict__ part = static_cast<AT *>(a.part);
    const int g = lane / G, li = lane % G;
    const bool has = g < tk.n;
    const int64_t item = tk.item0 + (has ? g : 0);
    const GramItem m = a.items[item - a.item0];
    const int cnt = has ? m.count : 0;
    // accumulators of this group width: in FP32 the entries rounded up to a multiple of G (the
    // reduce-scatter halves the set log2(G) times)
    constexpr bool FP64 = sizeof(AT) == 8;
    constexpr int NV = gram_nv(KT);
    constexpr int EPG = FP64 ? EP : (NV + G - 1) / G * G;
    AT acc[EPG];
#pragma unroll
    for (int v = 0; v < EPG; ++v) acc[v] = AT(0);
    // two observations per lane per iteration (lane order li, li+G, li+2G, ... is kept), so
    // that two gathers are in flight before either is consumed
    int e = li;
    for (; e + G < cnt; e += 2 * G) {
        const int64_t q0 = m.begin + e, q1 = q0 + G;
        const int c0 = __ldg(a.idx + q0), c1 = __ldg(a.idx + q1);
        const AT y0 = __ldg(val + q0), y1 = __ldg(val + q1);
        AT w0[KT], w1[KT];
        load_row<KT>(P + (int64_t)c0 * a.ldP, w0);
        load_row<KT>(P + (int64_t)c1 * a.ldP, w1);
        accum_all<KT, EPG, PART * EP, 0, AT>(acc, w0, y0);
        accum_all<KT, EPG, PART * EP, 0, AT>(acc, w1, y1);
    }
    if (e < cnt) {
        const int64_t q = m.begin + e;
        const int c = __ldg(a.idx + q);
        const AT y = __ldg(val + q);
        AT w[KT];
        load_row<KT>(P + (int64_t)c * a.ldP, w);
        accum_all<KT, EPG, PART * EP, 0, AT>(acc, w, y);
    }
    AT *dst = part + (item - a.item0) * (int64_t)a.ld + PART * EP;
    if constexpr (FP64) {
        int base = 0, end = NV - PART * EP < EP ? NV - PART * EP : EP;
        rs_uneven<EPG, G / 2, EPG, AT>(acc, lane, base, end);
        constexpr int PER = scattered<EPG, G / 2>();
#pragma unroll
        for (int v = 0; v < PER; ++v)
            if (has && base + v < end) dst[base + v] = acc[v];
    } else {
        rs_group<EPG, G / 2, EPG, AT>(acc, lane);
        constexpr int PER = EPG / G;
        if (has) {
#pragma unroll
            for (int v = 0; v < PER; ++v) dst[li * PER + v] = acc[v];
        }
    }
    if constexpr (G == 32) {
        // A row split over several items: the warp that completes the row's last item sums all
        // of the row's partials (FP64, item order) into the row's slot.  Publication order:
        // partial stores, fence, counter increment (no warp ever waits on another).
        const int mi = a.multi_idx[m.row];
        if (mi >= 0) {
            __threadfence();
            int last = 0;
            const int64_t r_i0 = a.item_ptr[m.row], r_i1 = a.item_ptr[m.row + 1];
            if (lane == 0) {
                const int old = atomicAdd(a.counters + (int64_t)mi * a.nparts + PART, 1);
                last = old == (int)(r_i1 - r_i0) - 1;
            }
            last = __shfl_sync(0xffffffffu, last, 0);
            if (last) {
                __threadfence();
                const int e1 = min((PART + 1) * EP, a.nv);
                for (int q = PART * EP + lane; q < e1; q += 32) {
                    double sum = 0.0;
                    for (int64_t it = r_i0; it < r_i1; ++it)
                        sum += (double)__ldcg(part + (it - a.item0) * (int64_t)a.ld + q);
                    a.rowsum[(int64_t)mi * a.ld_sum + q] = sum;
                }
                if (lane == 0) a.counters[(int64_t)mi * a.nparts + PART] = 0;
            }
        }
    }
}

template <int KT, typename GT, typename AT, int EP, int PART>
__device__ __forceinline__ void gram_body(const GramParams &a)
{
    const int lane = threadIdx.x & 31, wib = threadIdx.x >> 5;
    // warp by warp within a block; fewer tasks than warps go to different blocks instead, so that
    // they spread over the SMs
    const int64_t nwarps = ((int64_t)gridDim.x * blockDim.x) >> 5;
    const bool few = a.n_tasks < nwarps;
    for (int64_t t = few ? (int64_t)wib * gridDim.x + blockIdx.x : (int64_t)blockIdx.x * (blockDim.x >> 5) + wib;
         t < a.n_tasks; t += nwarps) {
        const GramTask tk = a.tasks[t];
        if (tk.G == 8)
            gram_task<KT, GT, AT, EP, PART, 8>(a, tk, lane);
        else if (tk.G == 16)
            gram_task<KT, GT, AT, EP, PART, 16>(a, tk, lane);
        else
            gram_task<KT, GT, AT, EP, PART, 32>(a, tk, lane);
    }
}

template <int KT, typename GT, typename AT, int EP, int PART, int NP>
__device__ __forceinline__ void gram_dispatch(int part, const GramParams &a)
{
    if constexpr (PART < NP) {
        if (part == PART)
            gram_body<KT, GT, AT, EP, PART>(a);
        else
            gram_dispatch<KT, GT, AT, EP, PART + 1, NP>(part, a);
    }
}

constexpr int kGramThreads = 256;

template <int KT, typename GT, typename AT, int EP>
__global__ void __launch_bounds__(kGramThreads, (EP > 96 ? 1 : 2)) gram_kernel(GramParams a)
{
    gram_dispatch<KT, GT, AT, EP, 0, parts_of(KT, sizeof(AT) == 8)>(blockIdx.y, a);
}

template <int KT, typename GT, typename AT>
static void launch_gram_t(const GramParams &a, int grid, cudaStream_t st)
{
    constexpr int EP = ep_of(KT, sizeof(AT) == 8);
    const dim3 g(grid, parts_of(KT, sizeof(AT) == 8));
    gram_kernel<KT, GT, AT, EP><<<g, kGramThreads, 0, st>>>(a);
}

template <int K, typename GT, typename AT>
static void launch_gram_k(const GramParams &a, int grid, cudaStream_t st)
{
    constexpr int KT = width_of(K, sizeof(AT) == 8);
    if (width_of(a.K, sizeof(AT) == 8) == KT)
        launch_gram_t<KT, GT, AT>(a, grid, st);
    else if constexpr (K > 1)
        launch_gram_k<K - 1, GT, AT>(a, grid, st);
}

void launch_gram(int prec, const GramParams &a, int grid, cudaStream_t st)
{
    if (a.n_tasks == 0) return;
    if (prec == BMF_FP64)
        launch_gram_k<16, double, double>(a, grid, st);
    else if (prec == BMF_FP32)
        launch_gram_k<16, float, float>(a, grid, st);
    else
        launch_gram_k<16, __nv_bfloat16, float>(a, grid, st);
}

}  // namespace bmf
