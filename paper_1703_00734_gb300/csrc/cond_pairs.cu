// cond_pairs.cu -- the conditional draw of every row given its partners for the reduced-precision
// modes (FP32, TF32 and BF16 gathers), in float pairs (fpair.cuh):
//   Lambda_n = Lambda_p + tau G_n,   b_n = Lambda_p mu_p + tau r_n,
//   Lambda_n = L L^T,  x_n = L^{-T} (L^{-1} b_n + z_n)
// (Eqs. 2-4, the (N+D)K^3 term of the cost model of Section 4.3), then the FP64 state, its
// gathered copy and the FP64 moment sums (Section 4.1).
//
// The FP64 pipe of this GPU takes a warp instruction every 17 clocks per SM; a multiply-add of
// float pairs is 12 FP32 instructions, 3.3 clocks, at 48 bits, where the Gram sums carry 24.
// Alone on the device, FP64 teams or threads per row before, this kernel now, per half sweep: K = 10,
// 69,878 rows 127 -> 91 us; K = 32, 120,047 rows 3,832 -> 1,184 us; K = 16, 225,000 rows with
// propagated priors and moment sums 1,221 -> 540 us for 163,000 of them and, beside it, 118 us for the
// others, which have no observations.  It issues 39 to 59% of the time: the pair arithmetic is about
// half of its 1,570 warp instructions per row at K = 16, the rest loads, splits and range checks.
//
// The dispatch: below K = 9 a row's FP64 work is small enough that a thread per row is as fast;
// above K = 48 the FP64 teams stay, because there a change in the last bit of a draw grows, through
// the FP32 gathers of ill-conditioned rows, to more than 2e-5 of the posterior means within ten
// sweeps (50,000 x 12,500, K = 64, sigma 0.3: 5e-5, half of what FP32 gathers are off by).
//
// Pairs stand in for FP64 only where the Gram sums' own rounding is what a row's draw is off by.  A
// row whose sums make up less than 2^-16 of every diagonal entry (above all a row without
// observations, which is its prior and its normals) is drawn in FP64.  Median error of a draw against
// 64-bit arithmetic on 64-bit partners at K = 16 with priors of condition 1e4, FP64 with its refined
// pivots for all rows / pairs for all rows / this: rows without observations 2.5e-13 / 1.4e-12 /
// 3.8e-14; with 1 to 15 observations 1.08e-7 (FP32) and 1.36e-3 (BF16), with 16 to 400 6.0e-8 and
// 4.6e-4, all three alike to three digits, as for K = 9 to 48.
//
// A row whose terms or results leave the range of a pair, or whose pivot loses 20 bits to
// cancellation (among them every row that is not positive definite), is redone in FP64 by a
// team, so what is accepted and what is rejected is decided in FP64.
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

__device__ __forceinline__ void decode_tri(int e, int &i, int &j)
{
    i = (int)((sqrtf(8.0f * e + 1.0f) - 1.0f) * 0.5f);
    while (i * (i + 1) / 2 > e) --i;
    while ((i + 1) * (i + 2) / 2 <= e) ++i;
    j = e - i * (i + 1) / 2;
}

// A pivot that lost 20 of its 48 bits (or is not positive, or NaN) sends its row to FP64.
constexpr float kPivotLoss = 0x1p-20f;
// The part of some diagonal entry that a row's sums must make up: their own rounding, 2^-24 of them, is
// then at least 2^-40 of the entry, 16 times a pair operation's 2^-44.
constexpr float kSumsShare = 0x1p-16f;

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

// What a row's Gram sums and prior are read from.
struct RowTerms {
    const double *ps, *pl, *pb;   // sums of several work items; prior precision and precision x mean
    const float *pp;              // one item's sums
    int64_t step;                 // between packed entries of the prior
    double tau;
    int mi;
    bool one;
    __device__ __forceinline__ RowTerms(const CondParams &a, int64_t r)
    {
        const int64_t i0 = a.item_ptr[r];
        const int h = a.row_hslot[r];
        mi = a.multi_idx[r];
        one = a.item_ptr[r + 1] > i0;
        tau = a.tau_row ? a.tau_row[r] : a.tau;
        const double *hp = a.hyper + (int64_t)(h >= 0 ? h : 0) * hyper_slot_len(a.K) + a.K;
        pl = h >= 0 ? hp : a.prior_L + r;
        pb = h >= 0 ? hp + ntri(a.K) : a.prior_b + r;
        step = h >= 0 ? 1 : a.R;
        ps = a.rowsum + (int64_t)(mi >= 0 ? mi : 0) * a.ld_sum;
        pp = static_cast<const float *>(a.part) + (i0 - a.item0) * (int64_t)a.ld;
    }
    __device__ __forceinline__ double sum(int e) const { return mi >= 0 ? ps[e] : (one ? widen(pp[e]) : 0.0); }
};

// State, gathered copy and moment sums of a drawn row (x in xd) by its team; the row's slots take the
// old moment sums.
template <int T, typename GT>
__device__ __forceinline__ void store_row(const CondParams &a, int64_t r, fpair *M, fpair *Y, const double *xd, int tl)
{
    const int K = a.K;
    const int64_t R = a.R;
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

// One row in FP64 by its team, x to xd.  False if a pivot is not positive.
//
// Four lanes (K <= 16): lane tl holds the rows tl + 4 s in registers; pivots and columns by shuffles.
template <int RMAX, typename GT>
__device__ __forceinline__ bool row_fp64_regs(const CondParams &a, int64_t r, fpair *M, fpair *Y, double *xd, int tl)
{
    constexpr int KP = 4 * RMAX;
    constexpr unsigned kFull = 0xffffffffu;
    const int K = a.K;
    const RowTerms t(a, r);
    const bool fused = t.mi == kFusedRow;
    if (fused) {
        Team<4, RMAX, GT> team{a, M, Y, nullptr, KP, tl, 0};
        team.own_gram(a.obs_ptr[r], (int)(a.obs_ptr[r + 1] - a.obs_ptr[r]));   // this lane's rows
    }
    double m[RMAX][KP], b[RMAX], x[RMAX];
#pragma unroll
    for (int s = 0; s < RMAX; ++s) {
        const int i = tl + 4 * s;
#pragma unroll
        for (int j = 0; j < KP; ++j)
            if (j < 4 * s + 4)
                m[s][j] = i < K && j <= i ? fma(t.tau, fused ? widen(M[row_off(i) + j].h) : t.sum(tri(i, j)),
                                                t.pl[(int64_t)tri(i, j) * t.step])
                                          : 0.0;
        b[s] = i < K ? fma(t.tau, fused ? widen(Y[i].h) : t.sum(a.part_rhs + i), t.pb[i * t.step]) : 0.0;
        x[s] = 0.0;
    }
    __syncwarp();
    bool ok = true;
#pragma unroll
    for (int k = 0; k < KP; ++k)
        if (k < K) {
            const double d = __shfl_sync(kFull, m[k / 4][k], k % 4, 4);
            ok = ok && pivot_ok(d);
            const double rs = ok ? rsqrt_full(d) : 0.0;
            const double y = __shfl_sync(kFull, b[k / 4], k % 4, 4) * rs;
            double l[RMAX];
#pragma unroll
            for (int s = 0; s < RMAX; ++s)
                if (s >= k / 4) {
                    l[s] = tl + 4 * s > k ? m[s][k] * rs : 0.0;
                    b[s] = fma(-l[s], y, b[s]);
                    m[s][k] = l[s];
                }
            if (tl == k % 4) {
                m[k / 4][k] = rs;   // 1 / L_kk in L_kk's place
                b[k / 4] = y;
            }
#pragma unroll
            for (int j = 0; j < KP; ++j)
                if (j > k) {
                    const double lj = __shfl_sync(kFull, l[j / 4], j % 4, 4);
#pragma unroll
                    for (int s = 0; s < RMAX; ++s)
                        if (s >= j / 4) m[s][j] = fma(-l[s], lj, m[s][j]);
                }
        }
    const double *z = a.z + (r - a.row0) * K;
#pragma unroll
    for (int s = 0; s < RMAX; ++s)
        if (tl + 4 * s < K) b[s] += z[tl + 4 * s];
    // x_i from the rows below it, each lane's share of them first (x[s] is zero until known)
#pragma unroll
    for (int i = KP - 1; i >= 0; --i)
        if (i < K) {
            double v = 0.0;
#pragma unroll
            for (int s = 0; s < RMAX; ++s)
                if (s >= i / 4) v = fma(m[s][i], x[s], v);
            v += __shfl_xor_sync(kFull, v, 1);
            v += __shfl_xor_sync(kFull, v, 2);
            if (tl == i % 4) x[i / 4] = (b[i / 4] - v) * m[i / 4][i];
        }
#pragma unroll
    for (int s = 0; s < RMAX; ++s)
        if (tl + 4 * s < K) xd[tl + 4 * s] = x[s];
    return ok;
}

// Wider teams: the row in the slots of its pairs (a slot is as long as a double), right-looking with the
// right-hand side as one more row, lane tl owning the rows tl + T s.
template <int T, int RMAX>
__device__ __forceinline__ bool row_fp64(const CondParams &a, int64_t r, double *M, double *Y, double *xd, int tl)
{
    const int K = a.K;
    const RowTerms t(a, r);
    for (int i = tl; i < K; i += T) {
        for (int j0 = 0; j0 <= i; j0 += 4) {
            double g[4], p[4];
#pragma unroll
            for (int u = 0; u < 4; ++u) {
                const int e = tri(i, min(j0 + u, i));
                g[u] = t.sum(e);
                p[u] = t.pl[(int64_t)e * t.step];
            }
#pragma unroll
            for (int u = 0; u < 4; ++u)
                if (j0 + u <= i) M[row_off(i) + j0 + u] = fma(t.tau, g[u], p[u]);
        }
        Y[i] = fma(t.tau, t.sum(a.part_rhs + i), t.pb[i * t.step]);
    }
    __syncwarp();
    bool ok = true;
    for (int k = 0, kk = 0; k < K; kk += 4 * (k >> 2) + 6, ++k) {   // kk: row_off(k)
        const double d = M[kk + k];
        ok = ok && pivot_ok(d);
        const double rs = ok ? rsqrt_full(d) : 0.0, y = Y[k] * rs;
        double l[RMAX];
#pragma unroll
        for (int s = 0; s < RMAX; ++s) {
            const int i = tl + T * s;
            l[s] = 0.0;
            if (i > k && i < K) M[row_off(i) + k] = l[s] = M[row_off(i) + k] * rs;
        }
        __syncwarp();
        if (tl == 0) M[kk + k] = rs, Y[k] = y;   // 1 / L_kk in L_kk's place
#pragma unroll
        for (int s = 0; s < RMAX; ++s) {
            const int i = tl + T * s;
            if (i > k && i < K) Y[i] = fma(-l[s], y, Y[i]);
        }
        for (int j = k + 1, jj = kk + 4 * (k >> 2) + 6; j < K; jj += 4 * (j >> 2) + 6, ++j) {
            const double lj = M[jj + k];
#pragma unroll
            for (int s = 0; s < RMAX; ++s) {
                const int i = tl + T * s;
                if (i >= j && i < K) M[row_off(i) + j] = fma(-l[s], lj, M[row_off(i) + j]);
            }
        }
        __syncwarp();
    }
    const double *z = a.z + (r - a.row0) * K;
    for (int i = tl; i < K; i += T) Y[i] += z[i];
    __syncwarp();
    for (int i = K - 1; i >= 0; --i) {
        const double *row = M + row_off(i);
        const double x = Y[i] * row[i];
        for (int k = tl; k < i; k += T) Y[k] = fma(-row[k], x, Y[k]);
        if (tl == 0) xd[i] = x;
        __syncwarp();
    }
    return ok;
}

// The rows row0 + (set bits of `rows`) of this CUDA block in FP64, a team each: those that pairs cannot
// hold, after the block's other rows.  They are dealt out anew, so that the teams of a warp (whose
// FP64 instructions cost the same whatever the active lanes) have one each, and stand apart from the
// pair draw, whose registers they would cost.  A lane alone on a row, where its team found it, waited
// on K^3 / 6 dependent operations: 60,000 rows of K / 2 observations and 20,000 ordinary ones, sigma =
// 0.002 to 0.003, where most rows lose their pivots' bits, us a sweep with FP64 teams or threads for
// all rows / pairs and a lane / pairs and these: K = 10 247 / 431 / 276, K = 16 487 / 2,035 / 594,
// K = 24 1,830 / 4,350 / 1,559 (ordinary noise: 250 / 185, 489 / 279, 1,744 / 677).
template <int T, int RMAX, typename GT>
__device__ __noinline__ void redo_rows(const CondParams &a, int64_t row0, unsigned long long rows, fpair *M, fpair *Y,
                                       double *xd, int tm, int tl, int n_teams)
{
    const int n = __popcll(rows);
    for (int base = 0; base < n; base += n_teams) {
        const bool mine = base + tm < n;
        if (!__any_sync(0xffffffffu, mine)) break;
        unsigned long long left = rows;      // teams without a row repeat the last one and drop it
        for (int q = min(base + tm, n - 1); q > 0; --q) left &= left - 1;
        const int64_t r = row0 + __ffsll((long long)left) - 1;
        __syncwarp();
        bool ok;
        if constexpr (T == 4)
            ok = row_fp64_regs<RMAX, GT>(a, r, M, Y, xd, tl);
        else
            ok = row_fp64<T, RMAX>(a, r, reinterpret_cast<double *>(M), reinterpret_cast<double *>(Y), xd, tl);
        __syncwarp();
        if (mine && ok) store_row<T, GT>(a, r, M, Y, xd, tl);
        if (mine && !ok && tl == 0) {
            atomicOr(&a.err->flags, ERR_NOT_PD);
            atomicMin(&a.err->first_bad_row, (int)r);
        }
        __syncwarp();
    }
}

// Rows without observations whose prior is their own (K <= kBareMaxK): nothing but their prior and their
// normals enters them, and no other row and no statistic waits for them.  x = L^{-T} (y + z) with
// L L^T = Lambda_p and L y = b_p, which stay as they are while a call's sweeps draw z: FP64, the factor
// once per call, the draws, K (K + 1) / 2 multiply-adds a row, beside the float pairs of the other rows.
// 225,000 rows at K = 16, 62,000 of them such rows, us a half sweep: 541 with pairs for all, 1,240
// with these drawn like redo_rows', 543 now.  (Above K = 16 redo_rows takes them: a thread's row no
// longer fits in registers.)
//
// The factor, a thread per row, the matrix interleaved in shared memory (entry e of a row at e * 32), four
// rows of a column at a time; out: [ntri(K) + K][n_all], entry by entry, 1 / L_jj on the diagonal (zero
// in entry 0 of a row that is not positive definite), then y.
__global__ void __launch_bounds__(32) bare_factor_kernel(const __grid_constant__ CondParams a, BareRows w)
{
    extern __shared__ double smd[];
    constexpr int W = 32, BATCH = 16;   // loads of a row in flight
    const int K = a.K, NT = ntri(K);
    double *A = smd + threadIdx.x;      // the packed triangle, then the right-hand side as its row K
    for (int64_t q = w.first + (int64_t)blockIdx.x * W + threadIdx.x; q < w.last; q += (int64_t)gridDim.x * W) {
        const int64_t r = w.rows[q];
        if (a.row_hslot[r] >= 0) continue;
        for (int e0 = 0; e0 < NT + K; e0 += BATCH) {
            double v[BATCH];
#pragma unroll
            for (int u = 0; u < BATCH; ++u) {
                const int e = min(e0 + u, NT + K - 1);
                v[u] = e < NT ? a.prior_L[(int64_t)e * a.R + r] : a.prior_b[(int64_t)(e - NT) * a.R + r];
            }
#pragma unroll
            for (int u = 0; u < BATCH; ++u)
                if (e0 + u < NT + K) A[(e0 + u) * W] = v[u];
        }
        bool ok = true;
        for (int j = 0; j < K; ++j) {
            double *Lj = A + tri(j, 0) * W;
            double d = Lj[j * W];
            for (int k = 0; k < j; ++k) d = fma(-Lj[k * W], Lj[k * W], d);
            ok = ok && pivot_ok(d);
            const double rs = ok ? rsqrt_full(d) : 0.0;
            Lj[j * W] = rs;
            for (int i0 = j + 1; i0 <= K; i0 += 4) {
                double *Li[4], v[4];
#pragma unroll
                for (int u = 0; u < 4; ++u) {
                    Li[u] = A + tri(min(i0 + u, K), 0) * W;
                    v[u] = Li[u][j * W];
                }
                for (int k = 0; k < j; ++k) {
                    const double l = Lj[k * W];
#pragma unroll
                    for (int u = 0; u < 4; ++u) v[u] = fma(-Li[u][k * W], l, v[u]);
                }
#pragma unroll
                for (int u = 0; u < 4; ++u)
                    if (i0 + u <= K) Li[u][j * W] = v[u] * rs;
            }
        }
        if (!ok) {
            atomicOr(&a.err->flags, ERR_NOT_PD);
            atomicMin(&a.err->first_bad_row, (int)r);
            A[0] = 0.0;
        }
        for (int e = 0; e < NT + K; ++e) w.factor[(int64_t)e * w.n_all + q] = A[e * W];
    }
}

// The draws, a thread per row: a row's factor, normals and moment sums once through memory.
template <int KM, typename GT>
__global__ void __launch_bounds__(128) bare_draw_kernel(const __grid_constant__ CondParams a, BareRows w)
{
    const int K = a.K, NT = ntri(K);
    const int64_t q = w.first + (int64_t)blockIdx.x * blockDim.x + threadIdx.x, N = w.n_all;
    if (q >= w.last) return;
    const int64_t r = w.rows[q];
    const double *F = w.factor + q;
    if (a.row_hslot[r] >= 0 || F[0] == 0.0) return;
    double x[KM];
    const double *z = a.z + (r - a.row0) * K;
#pragma unroll
    for (int i = 0; i < KM; ++i) x[i] = i < K ? F[(int64_t)(NT + i) * N] + z[i] : 0.0;
#pragma unroll
    for (int i = KM - 1; i >= 0; --i)
        if (i < K) {
            double l[KM];
#pragma unroll
            for (int k = 0; k <= i; ++k) l[k] = F[(int64_t)tri(i, k) * N];
            x[i] *= l[i];
#pragma unroll
            for (int k = 0; k < i; ++k) x[k] = fma(-l[k], x[i], x[k]);
        }
    GT *g = static_cast<GT *>(a.Xg) + r * a.ldg;
#pragma unroll
    for (int i = 0; i < KM; ++i)
        if (i < K) {
            a.X[r * K + i] = x[i];
            g[i] = gathered<GT>(x[i], (float)x[i]);
        }
    for (int i = K; i < a.ldg; ++i) g[i] = gathered<GT>(0.0, 0.f);
    if (!a.keep) return;
    double s[KM];
#pragma unroll
    for (int i = 0; i < KM; ++i) s[i] = a.S1[(int64_t)min(i, K - 1) * a.R + r];
#pragma unroll
    for (int i = 0; i < KM; ++i)
        if (i < K) a.S1[(int64_t)i * a.R + r] = s[i] + x[i];
    if (!a.full) return;
#pragma unroll
    for (int i = 0; i < KM; ++i)
        if (i < K) {
            double *S = a.S2 + (int64_t)tri(i, 0) * a.R + r;
#pragma unroll
            for (int j = 0; j <= i; ++j) s[j] = S[(int64_t)j * a.R];
#pragma unroll
            for (int j = 0; j <= i; ++j) S[(int64_t)j * a.R] = fma(x[i], x[j], s[j]);
        }
}

template <int T, int RMAX, typename GT>
__global__ void __launch_bounds__(256) cond_pairs_kernel(const __grid_constant__ CondParams a)
{
    extern __shared__ __align__(16) unsigned char smraw[];
    __shared__ unsigned long long redo_rest;   // rows of the block left for FP64
    __shared__ unsigned has[kCondBlock / 32];
    __shared__ uint8_t order[kCondBlock];
    const int K = a.K, NT = ntri(K), KP = padded4(K);
    const int lane = threadIdx.x & 31, tl = threadIdx.x % T, tm = threadIdx.x / T;
    const int n_teams = blockDim.x / T;
    fpair *M = reinterpret_cast<fpair *>(smraw) + (size_t)tm * team_pairs(K), *Y = M + row_off(KP);
    Team<T, RMAX, GT> team{a, M, Y, Y + KP, KP, tl, lane & ~(T - 1)};
    double *xd = reinterpret_cast<double *>(Y + 2 * KP);   // z, then the state
    const CondBlock blk = a.blocks[blockIdx.x];
    const int64_t R = a.R;
    // rows without observations are FP64's: the others are dealt to the block's parts and their teams
    // without gaps (30,011 x 2,027 at K = 24, 20 sweeps: 14.8 -> 13.7 to 14.7 ms)
    const int own = threadIdx.x;
    const bool sums_of = own < blk.n && a.item_ptr[blk.row0 + own + 1] > a.item_ptr[blk.row0 + own];
    if (own < kCondBlock) {
        const unsigned v = __ballot_sync(0xffffffffu, sums_of);
        if (lane == 0) has[own >> 5] = v;
    }
    __syncthreads();
    const unsigned long long with = (unsigned long long)has[1] << 32 | has[0];
    const int n_with = __popcll(with);
    if (sums_of) order[__popcll(with & ((1ull << own) - 1ull))] = (uint8_t)own;
    if (own == 0) {
        const bool apart = a.bare_apart && a.row_hslot[blk.row0] < 0;
        redo_rest = blockIdx.y > 0 || apart ? 0ull : ~with & (~0ull >> (kCondBlock - blk.n));
    }
    __syncthreads();
    const unsigned tmask = T == 32 ? 0xffffffffu : ((1u << T) - 1u) << (lane & ~(T - 1));
    const int rows = kCondBlock / gridDim.y, q_end = min(n_with, (int)(blockIdx.y + 1) * rows);
    for (int q0 = blockIdx.y * rows; q0 < q_end; q0 += n_teams) {
        const bool active = q0 + tm < q_end;
        const int q = active ? order[q0 + tm] : 0;
        const int64_t r = blk.row0 + q;
        bool bad = false, sums = false;
        // G, r and the prior (teams without a row carry an identity)
        if (active) {
            const int64_t i0 = a.item_ptr[r];
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
            } else {
                for (int i = tl; i < K; i += T) {
                    const float *src = pp + tri(i, 0);
                    fpair *dst = M + row_off(i);
                    for (int j = 0; j <= i; ++j) copy4(&dst[j].h, src + j);
                    copy4(&Y[i].h, pp + a.part_rhs + i);
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
                const float gd = M[row_off(i) + i].h;
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
                sums |= tau.h * gd >= kSumsShare * M[row_off(i) + i].h;
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
        const unsigned out = __ballot_sync(0xffffffffu, bad) & tmask, in = __ballot_sync(0xffffffffu, sums) & tmask;
        bool redo = out != 0u || in == 0u;
        if (__any_sync(0xffffffffu, active && !redo)) {
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
        }
        const unsigned lost = __ballot_sync(0xffffffffu, bad) & tmask;
        redo = redo || lost != 0u;
        __syncwarp();
        if (active && !redo) store_row<T, GT>(a, r, M, Y, xd, tl);
        if (active && redo && tl == 0) atomicOr(&redo_rest, 1ull << q);
        __syncwarp();
    }
    __syncthreads();
    if (redo_rest != 0ull) redo_rows<T, RMAX, GT>(a, blk.row0, redo_rest, M, Y, xd, tm, tl, n_teams);
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
    // us in parts; 225,000 rows: 660 and 609 us, all of them in pairs).
    auto bytes = [&](int th) { return (size_t)(th / T) * team_pairs(a.K) * sizeof(fpair); };
    auto fit = [&](int th) { return (int)std::min<size_t>(512 / th, (size_t)220 * 1024 / bytes(th)); };
    int threads = 256, parts = 1;
    while (threads > 64 && (threads / T > kCondBlock || n_blocks > sms * fit(threads))) threads /= 2;
    const int teams = threads / T;
    if (threads == 64)
        while (parts < kCondBlock / teams && (int64_t)n_blocks * parts < (int64_t)8 * sms * fit(threads)) parts *= 2;
    const size_t smem = bytes(threads);
    allow_smem(cond_pairs_kernel<T, RMAX, GT>, smem);
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
    if (prec == BMF_BF16)
        launch_pairs_t<__nv_bfloat16>(a, n_blocks, sms, st);
    else
        launch_pairs_t<float>(a, n_blocks, sms, st);
    return true;
}

void launch_bare_factor(const CondParams &a, const BareRows &w, int sms, cudaStream_t st)
{
    const size_t smem = (size_t)32 * (ntri(a.K) + a.K) * sizeof(double);   // 39 KB at K = 16: five per SM
    const int64_t blocks = std::min<int64_t>((int64_t)5 * sms, (w.last - w.first + 31) / 32);
    if (blocks > 0) bare_factor_kernel<<<(int)blocks, 32, smem, st>>>(a, w);
}

template <typename GT>
static void launch_draw_t(const CondParams &a, const BareRows &w, cudaStream_t st)
{
    const unsigned blocks = (unsigned)((w.last - w.first + 127) / 128);
    if (a.K <= 12)
        bare_draw_kernel<12, GT><<<blocks, 128, 0, st>>>(a, w);
    else
        bare_draw_kernel<kBareMaxK, GT><<<blocks, 128, 0, st>>>(a, w);
}

void launch_bare_draw(int prec, const CondParams &a, const BareRows &w, cudaStream_t st)
{
    if (w.last <= w.first) return;
    if (prec == BMF_BF16)
        launch_draw_t<__nv_bfloat16>(a, w, st);
    else
        launch_draw_t<float>(a, w, st);
}

}  // namespace bmf
