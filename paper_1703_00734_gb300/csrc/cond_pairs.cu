// cond_pairs.cu -- the conditional draw of every row given its partners for the reduced-precision
// modes (FP32, TF32 and BF16 gathers), in float pairs (fpair.cuh):
//   Lambda_n = Lambda_p + tau G_n,   b_n = Lambda_p mu_p + tau r_n,
//   Lambda_n = L L^T,  x_n = L^{-T} (L^{-1} b_n + z_n)
// (Eqs. 2-4, the (N+D)K^3 term of the cost model of Section 4.3), then the FP64 state, its
// gathered copy and the FP64 moment sums (Section 4.1).
//
// The FP64 pipe of this GPU takes a warp instruction every 17 clocks per SM; a multiply-add of
// float pairs is 12 FP32 instructions, 3.3 clocks, at 48 bits, where the Gram sums carry 24.
// Measured inside whole runs, FP64 teams or threads per row before, this kernel now, per half
// sweep: K = 16, 225,000 rows with propagated priors and moment sums 1,456 -> 855 us (617 us alone);
// K = 32, 120,047 rows 3,448 -> 1,409 us; K = 24, 30,011 rows 559 -> 240 us; K = 10, 69,878 rows
// 112 -> 95 us.  Alone it issues 47% of the time: the pair arithmetic is about half of its 1,440
// warp instructions per row at K = 16, the rest loads, splits and range checks.
//
// The dispatch: below K = 9 a row's FP64 work is small enough that a thread per row is as fast;
// above K = 48 the FP64 teams stay, because there a change in the last bit of a draw grows, through
// the FP32 gathers of ill-conditioned rows, to more than 2e-5 of the posterior means within ten
// sweeps (50,000 x 12,500, K = 64, sigma 0.3: 5e-5, half of what FP32 gathers are off by).
//
// A row whose terms leave the range of a pair, or whose pivot loses 20 bits to cancellation (among
// them every row that is not positive definite), is redone in FP64 by cond_row_serial, so what
// is accepted and what is rejected is decided in FP64.
#include <algorithm>

#include <cuda_bf16.h>

#include "common.cuh"
#include "fpair.cuh"
#include "kernels.h"

namespace bmf {

namespace {

template <typename GT>
__device__ __forceinline__ GT gathered(double x, float h);
template <>
__device__ __forceinline__ float gathered<float>(double, float h) { return h; }   // h = x rounded
template <>
__device__ __forceinline__ __nv_bfloat16 gathered<__nv_bfloat16>(double x, float) { return __double2bfloat16(x); }

__device__ __forceinline__ float as_float(float x) { return x; }
__device__ __forceinline__ float as_float(__nv_bfloat16 x) { return __bfloat162float(x); }

__device__ __forceinline__ void decode_tri(int e, int &i, int &j)
{
    i = (int)((sqrtf(8.0f * e + 1.0f) - 1.0f) * 0.5f);
    while (i * (i + 1) / 2 > e) --i;
    while ((i + 1) * (i + 2) / 2 <= e) ++i;
    j = e - i * (i + 1) / 2;
}

// One row in FP64 by one thread: S has room for ntri(K) + 2 K doubles; x is left at S + ntri(K).
// False (with the error word set) if a pivot is not positive.
template <typename GT>
__device__ __noinline__ bool cond_row_serial(const CondParams &a, int64_t r, double *S)
{
    const int K = a.K, NT = ntri(K);
    double *B = S + NT, *RI = B + K;
    const int64_t i0 = a.item_ptr[r], i1 = a.item_ptr[r + 1];
    const int mi = a.multi_idx[r], h = a.row_hslot[r];
    const double tau = a.tau_row ? a.tau_row[r] : a.tau;
    const double *hp = h >= 0 ? a.hyper + (int64_t)h * hyper_slot_len(K) : nullptr;
    for (int e = 0, i = 0, j = 0; e < NT + K; ++e) {
        // entry e: (i, j) of the packed lower triangle, then the right-hand side
        double g = 0.0;
        const int src = e < NT ? e : a.part_rhs + (e - NT);
        if (mi >= 0) {
            g = a.rowsum[(int64_t)mi * a.ld_sum + src];
        } else if (mi == kFusedRow) {
            float s = 0.f;
            for (int64_t o = a.obs_ptr[r]; o < a.obs_ptr[r + 1]; ++o) {
                const GT *p = static_cast<const GT *>(a.P) + (int64_t)a.obs_idx[o] * a.ldP;
                const float u = e < NT ? as_float(p[j]) : static_cast<const float *>(a.obs_val)[o];
                s = fmaf(as_float(p[e < NT ? i : e - NT]), u, s);
            }
            g = (double)s;
        } else if (i1 > i0) {
            g = (double)(static_cast<const float *>(a.part) + (i0 - a.item0) * (int64_t)a.ld)[src];
        }
        const double prior = e < NT ? (hp ? hp[K + e] : a.prior_L[(int64_t)e * a.R + r])
                                    : (hp ? hp[K + e] : a.prior_b[(int64_t)(e - NT) * a.R + r]);
        S[e] = fma(tau, g, prior);
        if (++j > i) ++i, j = 0;
    }
    for (int j = 0; j < K; ++j) {
        double d = S[tri(j, j)];
        for (int k = 0; k < j; ++k) d = fma(-S[tri(j, k)], S[tri(j, k)], d);
        if (!pivot_ok(d)) {
            atomicOr(&a.err->flags, ERR_NOT_PD);
            atomicMin(&a.err->first_bad_row, (int)r);
            return false;
        }
        const double rs = rsqrt(d);
        RI[j] = rs;
        for (int i = j + 1; i < K; ++i) {
            double s = S[tri(i, j)];
            for (int k = 0; k < j; ++k) s = fma(-S[tri(i, k)], S[tri(j, k)], s);
            S[tri(i, j)] = s * rs;
        }
    }
    for (int i = 0; i < K; ++i) {
        double s = B[i];
        for (int k = 0; k < i; ++k) s = fma(-S[tri(i, k)], B[k], s);
        B[i] = s * RI[i];
    }
    const double *z = a.z + (r - a.row0) * K;
    for (int i = K - 1; i >= 0; --i) {
        double s = B[i] + z[i];
        for (int k = i + 1; k < K; ++k) s = fma(-S[tri(k, i)], B[k], s);
        B[i] = s * RI[i];
    }
    return true;
}

// A pivot that lost 20 of its 48 bits (or is not positive, or NaN) sends its row to FP64.
constexpr float kPivotLoss = 0x1p-20f;

}  // namespace

// ------------------------------------------------------------------------------------------
// A team of T lanes per row, the row's matrix as pairs in shared memory, factored left-looking in
// panels of four columns: a lane holds the panel entries of up to RMAX rows in registers, takes
// the inner products with the finished columns (per two columns one 16-byte load per row and
// four shared by the team for 8 multiply-adds per row), factors the panel with shuffles and
// writes it back.  The forward solve rides along: the lane of panel row i also accumulates
// b_i - sum_k L_ik y_k.  The back solve goes panel by panel, its 4 x 4 triangle in every lane.
//
// Between the matrix operations the kernel waits for memory (a row's prior and moment sums are
// 2.4 KB at K = 16), so its loads go out together: the Gram sums and, after the draw, the moment
// sums are copied by cp.async into the matrix slots (a slot is a pair, as long as a double), the
// prior is read four entries ahead.  The loops are rolled where they can be: unrolled they
// outgrow the instruction cache.
//
// Row i is stored 4 (i / 4 + 1) + 2 pairs long, so that the rows of a panel are an odd number of
// 16-byte units apart: the four rows of a team and the neighbouring team's (half a bank cycle on)
// read without bank conflicts.  K is padded to a multiple of four with an identity.
// ------------------------------------------------------------------------------------------
__host__ __device__ constexpr int row_off(int i)
{
    return 8 * (i >> 2) * ((i >> 2) + 2) + (i & 3) * (4 * (i >> 2) + 6);
}
__host__ __device__ constexpr int padded4(int K) { return (K + 3) / 4 * 4; }
// pairs per team: the matrix, y, the reciprocal pivots, z / the state; 8 modulo 16 pairs (64
// bytes modulo a bank cycle)
__host__ __device__ constexpr int team_pairs(int K)
{
    return (row_off(padded4(K)) + 3 * padded4(K) + 7) / 16 * 16 + 8;
}

// A lane copies only what it reads back itself: its own wait is enough.
__device__ __forceinline__ void copy8(void *dst, const double *src)
{
    const unsigned d = (unsigned)__cvta_generic_to_shared(dst);
    asm volatile("cp.async.ca.shared.global [%0], [%1], 8;\n" ::"r"(d), "l"(src) : "memory");
}
__device__ __forceinline__ void copy4(float *dst, const float *src)
{
    const unsigned d = (unsigned)__cvta_generic_to_shared(dst);
    asm volatile("cp.async.ca.shared.global [%0], [%1], 4;\n" ::"r"(d), "l"(src) : "memory");
}
__device__ __forceinline__ void copies_wait() { asm volatile("cp.async.wait_all;\n" ::: "memory"); }

template <int T, int RMAX, typename GT>
struct Team {
    const CondParams &a;
    fpair *M, *Y, *RI;
    int KP, tl, base;   // padded K, lane of the team, its first lane of the warp

    __device__ __forceinline__ static float4 two(const fpair *p) { return *reinterpret_cast<const float4 *>(p); }

    // Columns p .. p + 3 with R rows per lane (rows p + tl + T s).  Returns false in the lane whose
    // pivot fails.
    template <int R>
    __device__ __forceinline__ bool panel(int p)
    {
        fpair acc[R][4], accy = fpair{0.f, 0.f};
        const fpair *row[R];
#pragma unroll
        for (int s = 0; s < R; ++s) {
            const int i = p + tl + T * s;
            row[s] = M + row_off(i < KP ? i : p);   // lanes past the last row repeat row p
#pragma unroll
            for (int c = 0; c < 4; c += 2) {
                const float4 v = two(row[s] + p + c);
                acc[s][c] = fpair{v.x, v.y};
                acc[s][c + 1] = fpair{v.z, v.w};
            }
        }
        if (tl < 4) accy = Y[p + tl];
        const float full = tl == 0 ? acc[0][0].h : tl == 1 ? acc[0][1].h : tl == 2 ? acc[0][2].h : acc[0][3].h;
        const fpair *col[4];
#pragma unroll
        for (int c = 0; c < 4; ++c) col[c] = M + row_off(p + c);
        for (int k = 0; k < p; k += 2) {
            float4 cv[4];
#pragma unroll
            for (int c = 0; c < 4; ++c) cv[c] = two(col[c] + k);
            const float4 yv = two(Y + k);
#pragma unroll
            for (int s = 0; s < R; ++s) {
                const float4 o = two(row[s] + k);
#pragma unroll
                for (int c = 0; c < 4; ++c) {
                    acc[s][c] = pfnma(acc[s][c], fpair{o.x, o.y}, fpair{cv[c].x, cv[c].y});
                    acc[s][c] = pfnma(acc[s][c], fpair{o.z, o.w}, fpair{cv[c].z, cv[c].w});
                }
                if (s == 0) {
                    accy = pfnma(accy, fpair{o.x, o.y}, fpair{yv.x, yv.y});
                    accy = pfnma(accy, fpair{o.z, o.w}, fpair{yv.z, yv.w});
                }
            }
        }
        bool good = true;
#pragma unroll
        for (int c = 0; c < 4; ++c) {
            const fpair d = shfl_pair(renorm(acc[0][c]), base + c);
            if (tl == c) good = pair_diag(full) && d.h >= full * kPivotLoss;
            const fpair rs = prsqrt(d);
            const fpair yc = shfl_pair(pmul(renorm(accy), rs), base + c);
            if (tl == c) {
                RI[p + c] = rs;
                Y[p + c] = yc;
            }
#pragma unroll
            for (int s = 0; s < R; ++s) acc[s][c] = pmul(renorm(acc[s][c]), rs);
            accy = pfnma(accy, acc[0][c], yc);
#pragma unroll
            for (int c2 = c + 1; c2 < 4; ++c2) {
                const fpair l = shfl_pair(acc[0][c], base + c2);
#pragma unroll
                for (int s = 0; s < R; ++s) acc[s][c2] = pfnma(acc[s][c2], acc[s][c], l);
            }
        }
#pragma unroll
        for (int s = 0; s < R; ++s) {
            const int i = p + tl + T * s;
            if (i < KP) {
                float4 *q = reinterpret_cast<float4 *>(M + row_off(i) + p);
                q[0] = make_float4(acc[s][0].h, acc[s][0].l, acc[s][1].h, acc[s][1].l);
                q[1] = make_float4(acc[s][2].h, acc[s][2].l, acc[s][3].h, acc[s][3].l);
            }
        }
        __syncwarp();
        return good;
    }

    // Panels whose row count needs R rows per lane, then those that need fewer.
    template <int R>
    __device__ __forceinline__ bool factor(int p)
    {
        bool good = true;
        for (; p < KP && KP - p > (R - 1) * T; p += 4) good = panel<R>(p) && good;
        if constexpr (R > 1) good = factor<R - 1>(p) && good;
        return good;
    }

    // x = L^{-T} Y in place.
    __device__ __forceinline__ void back()
    {
        for (int p = KP - 4; p >= 0; p -= 4) {
            fpair v[4], x[4];
#pragma unroll
            for (int c = 0; c < 4; ++c) v[c] = Y[p + c];
#pragma unroll
            for (int c = 3; c >= 0; --c) {
                x[c] = pmul(renorm(v[c]), RI[p + c]);
#pragma unroll
                for (int b = 0; b < c; ++b) v[b] = pfnma(v[b], M[row_off(p + c) + p + b], x[c]);
            }
            __syncwarp();
            if (tl < 4) Y[p + tl] = tl == 0 ? x[0] : tl == 1 ? x[1] : tl == 2 ? x[2] : x[3];
            for (int k = tl; k < p; k += T) {
                fpair s = Y[k];
#pragma unroll
                for (int c = 3; c >= 0; --c) s = pfnma(s, M[row_off(p + c) + k], x[c]);
                Y[k] = s;
            }
            __syncwarp();
        }
    }

    // Gram sums of a row with few observations (13 <= K <= 16), in list order, FP32: rows tl + 4 s
    // of the packed triangle in this lane.
    __device__ __forceinline__ void own_gram(int64_t o0, int no)
    {
        float G[RMAX][4 * RMAX], Rv[RMAX];
#pragma unroll
        for (int s = 0; s < RMAX; ++s) {
            Rv[s] = 0.f;
#pragma unroll
            for (int j = 0; j < 4 * s + 4; ++j) G[s][j] = 0.f;
        }
        constexpr int QG = 4;   // indices and values of four observations, then their rows
        for (int c0 = 0; c0 < no; c0 += QG) {
            int32_t pid[QG];
            float yv[QG];
#pragma unroll
            for (int q = 0; q < QG; ++q) {
                const bool in = c0 + q < no;
                pid[q] = in ? __ldg(a.obs_idx + o0 + c0 + q) : 0;
                yv[q] = in ? __ldg(static_cast<const float *>(a.obs_val) + o0 + c0 + q) : 0.f;
            }
#pragma unroll
            for (int q = 0; q < QG; ++q)
                if (c0 + q < no) {
                    const GT *pr = static_cast<const GT *>(a.P) + (int64_t)pid[q] * a.ldP;
                    float pv[4 * RMAX];
                    if constexpr (sizeof(GT) == 4) {
#pragma unroll
                        for (int c = 0; c < RMAX; ++c) {
                            const float4 v = __ldg(reinterpret_cast<const float4 *>(pr) + c);
                            pv[4 * c] = v.x, pv[4 * c + 1] = v.y, pv[4 * c + 2] = v.z, pv[4 * c + 3] = v.w;
                        }
                    } else {
#pragma unroll
                        for (int c = 0; c < RMAX; ++c) {
                            const uint2 v = __ldg(reinterpret_cast<const uint2 *>(pr) + c);
                            pv[4 * c] = __uint_as_float(v.x << 16), pv[4 * c + 1] = __uint_as_float(v.x & 0xffff0000u);
                            pv[4 * c + 2] = __uint_as_float(v.y << 16), pv[4 * c + 3] = __uint_as_float(v.y & 0xffff0000u);
                        }
                    }
#pragma unroll
                    for (int s = 0; s < RMAX; ++s) {
                        const float own = tl == 0 ? pv[4 * s] : tl == 1 ? pv[4 * s + 1] : tl == 2 ? pv[4 * s + 2] : pv[4 * s + 3];
#pragma unroll
                        for (int j = 0; j < 4 * s + 4; ++j) G[s][j] = fmaf(own, pv[j], G[s][j]);
                        Rv[s] = fmaf(yv[q], own, Rv[s]);
                    }
                }
        }
#pragma unroll
        for (int s = 0; s < RMAX; ++s) {
            fpair *q = M + row_off(4 * s) + tl * (4 * s + 6);
#pragma unroll
            for (int j = 0; j < 4 * s + 4; ++j) q[j].h = G[s][j];
            Y[tl + 4 * s].h = Rv[s];
        }
    }
};

template <int T, int RMAX, typename GT>
__global__ void __launch_bounds__(256) cond_pairs_kernel(const __grid_constant__ CondParams a)
{
    extern __shared__ __align__(16) unsigned char smraw[];
    const int K = a.K, NT = ntri(K), KP = padded4(K);
    const int lane = threadIdx.x & 31, tl = threadIdx.x % T, tm = threadIdx.x / T;
    const int n_teams = blockDim.x / T;
    fpair *M = reinterpret_cast<fpair *>(smraw) + (size_t)tm * team_pairs(K), *Y = M + row_off(KP);
    Team<T, RMAX, GT> team{a, M, Y, Y + KP, KP, tl, lane & ~(T - 1)};
    double *xd = reinterpret_cast<double *>(Y + 2 * KP);   // z, then the state
    const CondBlock blk = a.blocks[blockIdx.x];
    const int64_t R = a.R;
    const unsigned tmask = T == 32 ? 0xffffffffu : ((1u << T) - 1u) << (lane & ~(T - 1));
    const int rows = kCondBlock / gridDim.y, q_end = min(blk.n, (int)(blockIdx.y + 1) * rows);
    for (int q0 = blockIdx.y * rows; q0 < q_end; q0 += n_teams) {
        const int q = q0 + tm;
        const bool active = q < q_end;
        const int64_t r = blk.row0 + (active ? q : 0);
        bool bad = false;
        // G, r and the prior (teams past the block's rows carry an identity)
        if (active) {
            const int64_t i0 = a.item_ptr[r], i1 = a.item_ptr[r + 1];
            const int mi = a.multi_idx[r], h = a.row_hslot[r];
            const double tau_d = a.tau_row ? a.tau_row[r] : a.tau;
            const int64_t o0 = T == 4 ? a.obs_ptr[r] : 0, o1 = T == 4 ? a.obs_ptr[r + 1] : 0;
            const double *hp = a.hyper + (int64_t)(h >= 0 ? h : 0) * hyper_slot_len(K) + K;
            const double *pl = h >= 0 ? hp : a.prior_L + r, *pb = h >= 0 ? hp + NT : a.prior_b + r;
            const int64_t step = h >= 0 ? 1 : R;   // between packed entries of the prior
            const double *z = a.z + (r - a.row0) * K;
            for (int i = tl; i < K; i += T) copy8(xd + i, z + i);
            // the Gram sums into the slots of this lane's rows i = tl + T s
            const float *pp = static_cast<const float *>(a.part) + (i0 - a.item0) * (int64_t)a.ld;
            const bool exact = mi >= 0;            // FP64 sums: the slots' low parts count
            if (exact) {
                // a row split over several work items
                const double *ps = a.rowsum + (int64_t)mi * a.ld_sum;
                for (int i = tl; i < K; i += T)
#pragma unroll 4
                    for (int j = 0; j <= i + 1; ++j) {
                        const double g = ps[j <= i ? tri(i, j) : a.part_rhs + i];
                        bad |= !pair_below(g);
                        (j <= i ? M[row_off(i) + j] : Y[i]) = split(g);
                    }
            } else if (T == 4 && mi == kFusedRow) {
                if constexpr (T == 4) team.own_gram(o0, (int)(o1 - o0));
            } else if (i1 > i0) {
                for (int i = tl; i < K; i += T) {
                    const float *src = pp + tri(i, 0);
                    fpair *dst = M + row_off(i);
                    for (int j = 0; j <= i; ++j) copy4(&dst[j].h, src + j);
                    copy4(&Y[i].h, pp + a.part_rhs + i);
                }
            } else {
                for (int i = tl; i < K; i += T) {
                    for (int j = 0; j <= i; ++j) M[row_off(i) + j].h = 0.f;
                    Y[i].h = 0.f;
                }
            }
            // prior + tau g, four entries at a time, the next four priors in flight
            bad |= !pair_vector(tau_d);
            const fpair tau = split(tau_d);
            auto assemble = [&](fpair *slot, double p) {
                const fpair g{slot->h, exact ? slot->l : 0.f};
                bad |= !pair_below(p) | !(fabsf(g.h) < 0x1p70f);
                *slot = passemble(split(p), tau, g);
            };
            copies_wait();
            double nxt[4];
#pragma unroll
            for (int u = 0; u < 4; ++u) nxt[u] = tl < K ? pl[(int64_t)tri(tl, min(u, tl)) * step] : 0.0;
            for (int i = tl; i < K; i += T) {
                const double pr = pb[i * step];
                for (int j0 = 0; j0 <= i; j0 += 4) {
                    double cur[4];
#pragma unroll
                    for (int u = 0; u < 4; ++u) cur[u] = nxt[u];
                    const int ni = j0 + 4 <= i ? i : i + T, nj = j0 + 4 <= i ? j0 + 4 : 0;
                    if (ni < K)
#pragma unroll
                        for (int u = 0; u < 4; ++u) nxt[u] = pl[(int64_t)tri(ni, min(nj + u, ni)) * step];
#pragma unroll
                    for (int u = 0; u < 4; ++u)
                        if (j0 + u <= i) assemble(M + row_off(i) + j0 + u, cur[u]);
                }
                // the terms and their sum: tau g alone can leave FP32's exponents
                const float g = Y[i].h;
                assemble(Y + i, pr);
                bad |= !pair_vector(pr) | !pair_vector(Y[i].h) | (Y[i].h == 0.f && g != 0.f);
            }
        }
        for (int i = active ? K + tl : tl; i < KP; i += T) {
            for (int j = 0; j <= i; ++j) M[row_off(i) + j] = fpair{i == j ? 1.f : 0.f, 0.f};
            Y[i] = fpair{0.f, 0.f};
        }
        __syncwarp();
        bad |= !team.template factor<RMAX>(0);
        for (int i = tl; i < K && active; i += T) {
            const double zi = xd[i];
            Y[i] = padd(Y[i], split(zi));
            bad |= !pair_vector(zi) | !pair_vector(Y[i].h);
        }
        __syncwarp();
        team.back();
        for (int i = tl; i < K; i += T) {
            const fpair x = renorm(Y[i]);
            bad |= !pair_vector(x.h);
            xd[i] = join(x);
        }
        bool ok = active;
        const bool redo = (__ballot_sync(0xffffffffu, bad) & tmask) != 0u;
        if (active && redo) {
            int done = 0;
            if (tl == 0) done = cond_row_serial<GT>(a, r, reinterpret_cast<double *>(M)) ? 1 : 0;
            ok = __shfl_sync(tmask, done, lane & ~(T - 1)) != 0;
            __syncwarp(tmask);
            for (int i = tl; i < K; i += T) xd[i] = reinterpret_cast<double *>(M)[NT + i];
        }
        __syncwarp();
        // state, gathered copy, moment sums
        if (ok) {
            if (a.keep) {
                for (int i = tl; i < K; i += T) {
                    copy8(Y + i, a.S1 + (int64_t)i * R + r);
                    if (a.full) {
                        const double *src = a.S2 + (int64_t)tri(i, 0) * R + r;
                        fpair *dst = M + row_off(i);
                        for (int j = 0; j <= i; ++j) copy8(dst + j, src + j * R);
                    }
                }
            }
            GT *g = static_cast<GT *>(a.Xg) + r * a.ldg;
            for (int i = tl; i < K; i += T) {
                const double xi = xd[i];
                a.X[r * K + i] = xi;
                g[i] = gathered<GT>(xi, (float)xi);
            }
            for (int i = K + tl; i < a.ldg; i += T) g[i] = gathered<GT>(0.0, 0.f);
            if (a.keep) {
                copies_wait();
                for (int i = tl; i < K; i += T) {
                    const double xi = xd[i];
                    a.S1[(int64_t)i * R + r] = *reinterpret_cast<const double *>(Y + i) + xi;
                    if (a.full) {
                        double *dst = a.S2 + (int64_t)tri(i, 0) * R + r;
                        const fpair *src = M + row_off(i);
#pragma unroll 4
                        for (int j = 0; j <= i; ++j)
                            dst[j * R] = fma(xi, xd[j], *reinterpret_cast<const double *>(src + j));
                    }
                }
            }
        }
        __syncwarp();
    }
    // per-block statistics of the new state for the next hyperparameter draw (only blocks whose
    // factor draws its hyperparameters: every row of a block shares its subset's prior), read back
    // from the state rows this block has just written, each entry over the rows in order
    if (a.stats == nullptr || a.row_hslot[blk.row0] < 0) return;
    if (!last_part(a.parts_done, a.blk0 + blockIdx.x, gridDim.y)) return;
    const int NS = K + NT;
    const double *Xb = a.X + blk.row0 * K;
    double *out = a.stats + (a.blk0 + blockIdx.x) * (int64_t)NS;
    for (int e = threadIdx.x; e < NS; e += blockDim.x) {
        double s = 0.0;
        if (e < K) {
            for (int qq = 0; qq < blk.n; ++qq) s += __ldcg(Xb + qq * K + e);
        } else {
            int i, j;
            decode_tri(e - K, i, j);
            for (int qq = 0; qq < blk.n; ++qq) s = fma(__ldcg(Xb + qq * K + i), __ldcg(Xb + qq * K + j), s);
        }
        out[e] = s;
    }
}

template <int T, int RMAX, typename GT>
static void launch_team_t(const CondParams &a, int n_blocks, int sms, cudaStream_t st)
{
    // A launch whose conditional blocks fit on the GPU at once takes the widest CUDA blocks that do:
    // the rows go over more warps, and the block's statistics over more threads (K = 10, 10,677
    // rows: 63 us with 64 threads, 32 us with 256).  Larger launches take 64 threads, which fill an
    // SM evenly, and the rows of a conditional block in as many parts as rounds of its teams, until
    // the launch fills the GPU about eight times over (K = 16, 45,000 rows: 245 us as one part, 149
    // us in parts; 225,000 rows: 660 and 609 us).
    auto bytes = [&](int th) { return (size_t)(th / T) * team_pairs(a.K) * sizeof(fpair); };
    auto fit = [&](int th) { return (int)std::min<size_t>(512 / th, (size_t)220 * 1024 / bytes(th)); };
    int threads = 256, parts = 1;
    while (threads > 64 && (threads / T > kCondBlock || n_blocks > sms * fit(threads))) threads /= 2;
    const int teams = threads / T;
    if (threads == 64)
        while (parts < kCondBlock / teams && (int64_t)n_blocks * parts < (int64_t)8 * sms * fit(threads)) parts *= 2;
    const size_t smem = bytes(threads);
    if (smem > 48 * 1024)
        cudaFuncSetAttribute(cond_pairs_kernel<T, RMAX, GT>, cudaFuncAttributeMaxDynamicSharedMemorySize, (int)smem);
    cond_pairs_kernel<T, RMAX, GT><<<dim3(n_blocks, parts), threads, smem, st>>>(a);
}

template <typename GT>
static void launch_pairs_t(const CondParams &a, int n_blocks, int sms, cudaStream_t st)
{
    if (a.K <= 12)
        launch_team_t<4, 3, GT>(a, n_blocks, sms, st);
    else if (a.K <= 16)
        launch_team_t<4, 4, GT>(a, n_blocks, sms, st);
    else if (a.K <= 24)
        launch_team_t<8, 3, GT>(a, n_blocks, sms, st);
    else if (a.K <= 32)
        launch_team_t<8, 4, GT>(a, n_blocks, sms, st);
    else
        launch_team_t<16, 3, GT>(a, n_blocks, sms, st);
}

bool launch_cond_pairs(int prec, const CondParams &a, int n_blocks, int sms, cudaStream_t st)
{
    if (prec == BMF_FP64 || a.K < kPairsMinK || a.K > kPairsMaxK) return false;
    if (n_blocks <= 0) return true;
    if (prec == BMF_FP32)
        launch_pairs_t<float>(a, n_blocks, sms, st);
    else
        launch_pairs_t<__nv_bfloat16>(a, n_blocks, sms, st);
    return true;
}

}  // namespace bmf
