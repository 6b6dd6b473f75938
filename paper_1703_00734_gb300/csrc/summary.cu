// summary.cu -- the subset-posterior summaries beyond moment matching (Section 4.1, "PP DM"
// and "PP GMM"; Section 5.1) and the component choice of a propagated mixture prior.
//
//   * cluster_kernel: one warp per row clusters the row's retained samples by lambda-means and
//     forms the means and covariances of the largest clusters (dominant mode: the largest one;
//     mixture: the C largest with at least K + 1 samples, weighted by their sizes);
//   * fit_kernel: one thread per row takes their precisions (a row without such a cluster falls
//     back to one Gaussian over all samples) and the mixture's pooled mean and covariance, which
//     Eq. 14 aggregates (Section 4.2).  20,000 rows of 200 samples at K = 10, three modes:
//     21.0 ms with one warp per row for everything, 2.2 ms with these;
//   * mix_choose_kernel: one thread per row picks, before each draw, the component with the
//     largest responsibility pi_c N(x; mu_c, Lambda_c^{-1}) at the row's current value and
//     installs it as the row's prior.
//
// lambda-means follows one fixed procedure (the paper names the method without its details):
// one cluster centred on the first sample; each round visits the samples in order and gives
// each to the nearest centre (lowest index on ties) unless every squared distance exceeds
// lambda, in which case it opens a new cluster centred on itself; then centres move to the
// means of their samples and empty clusters are dropped (renumbered in order); rounds repeat
// until no assignment changes (at most 100).  The warp scores the samples in parallel against
// the existing centres, then walks the samples in order to open new clusters, updating the
// later samples' nearest centre after each opening: the same assignments as the sequential
// visit.  Every sum runs over the samples in order, so assignments and fits do not depend on the
// launch shape.
#include <algorithm>
#include <cmath>

#include "common.cuh"
#include "kernels.h"
#include "rows.cuh"

namespace bmf {

namespace {

constexpr unsigned kAll = 0xffffffffu;

__device__ __forceinline__ double dmul(double a, double b) { return __dmul_rn(a, b); }
__device__ __forceinline__ double dadd(double a, double b) { return __dadd_rn(a, b); }
__device__ __forceinline__ double dsub(double a, double b) { return __dsub_rn(a, b); }

// Squared distance of two K-vectors, summed in order.
__device__ double sqdist(const double *p, const double *c, int K)
{
    double d = 0.0;
    for (int k = 0; k < K; ++k) {
        const double e = dsub(p[k], c[k]);
        d = dadd(d, dmul(e, e));
    }
    return d;
}

// The same in FP32 from rounded vectors.
__device__ float sqdist32(const float *p, const float *c, int K)
{
    float d = 0.f;
    for (int k = 0; k < K; ++k) {
        const float e = p[k] - c[k];
        d = fmaf(e, e, d);
    }
    return d;
}

// Where the fits of a row pass between the two kernels: sizes, means and packed lower covariances
// of up to C components, inside the arrays that end up holding the results.  Row index q is
// row - row0 (fit outputs) or the arena row (library layout).
struct FitStage {
    double *n, *m, *S;
    int64_t n_row, n_c, m_row, m_c, S_row, S_c, S_e;
    __device__ double &size(int64_t q, int c) const { return n[q * n_row + c * n_c]; }
    __device__ double &mean(int64_t q, int c, int k) const { return m[q * m_row + c * m_c + k]; }
    __device__ double &cov(int64_t q, int c, int e) const { return S[q * S_row + c * S_c + e * S_e]; }
};

__host__ __device__ FitStage fit_stage(const SummaryParams &p)
{
    const int64_t K = p.K, C = p.C, KK = K * K, W = 1 + 2 * K + K * (K + 1) / 2;
    if (p.pi) return FitStage{p.pi, p.mu, p.Lam, C, 1, C * K, K, C * KK, KK, 1};
    if (p.mix) return FitStage{p.mix, p.mix + 1, p.mix + 1 + K, C * W, W, C * W, W, C * W, W, 1};
    return FitStage{p.mm_b, p.mm_mu, p.mm_L, 1, 0, K, 0, 1, 0, p.R};   // one component
}

constexpr int kFastCentres = 32;

// Shared memory of one row (one warp) with at most `cap` clusters at a time (S of them survive a
// round); fast: with FP32 copies of samples and centres.
size_t cluster_smem(int K, int S, int cap, bool fast)
{
    const size_t centres = (size_t)std::min(cap, std::max(S, 1));
    return ((size_t)S + centres) * K * (sizeof(double) + (fast ? sizeof(float) : 0)) +
           (size_t)S * (sizeof(float) + 4 * sizeof(int)) + (2 * (size_t)cap + centres + 1) * sizeof(int);
}

}  // namespace

// lambda-means of one row per warp and the covariances of its chosen clusters.  FAST rows keep at
// most `cap` clusters; rows that open more are listed for a second launch with room for
// every sample's own (2 S + 1 within a round: a centre opened in the round is its sample).
//
// The distances decide only comparisons (which centre is nearest, whether it is beyond lambda):
// FAST takes them in FP32, and again in FP64 where the FP32 values are closer than their error
// bound, so the assignments are those of the FP64 procedure at a fraction of its FP64 work (a
// warp's FP64 instruction takes 17 clocks of an SM, an FP32 one a quarter).  Centre means and
// covariances run over member lists in sample order.
template <bool FAST>
__global__ void __launch_bounds__(32) cluster_kernel(SummaryParams p, int cap, const int32_t *list,
                                                     const int32_t *list_n, int32_t *over, int32_t *over_n)
{
    extern __shared__ double sh[];
    const int lane = threadIdx.x;
    const int K = p.K, S = p.S, C = p.C, NT = K * (K + 1) / 2, centres = min(cap, max(S, 1));
    double *X = sh;                                              // [S][K]
    double *cen = X + (size_t)S * K;                             // [centres][K]
    float *Xf = reinterpret_cast<float *>(cen + (size_t)centres * K);   // [S][K] (FAST)
    float *cenf = Xf + (FAST ? (size_t)S * K : 0);               // [centres][K] (FAST)
    float *dbf = cenf + (FAST ? (size_t)centres * K : 0);        // [S] FP32 distance to the nearest
    int *assign = reinterpret_cast<int *>(dbf + S);              // [S]
    int *prev = assign + S;                                      // [S]
    int *far = prev + S;                                         // [S] nearest is beyond lambda
    int *member = far + S;                                       // [S] samples by cluster, in order
    int *opened = member;                                        // before that: samples of the round's new centres
    int *cnt = member + S, *map = cnt + cap, *off = map + cap;   // [cap], [cap], [centres + 1]
    const FitStage fs = fit_stage(p);
    const int64_t n_work = list ? (int64_t)*list_n : p.n_rows;
    for (int64_t w = blockIdx.x; w < n_work; w += gridDim.x) {
        const int64_t row = list ? list[w] : w;
        __syncwarp();
        float big = 0.f;
        for (int e = lane; e < S * K; e += 32) {
            const int s = e / K, k = e % K;
            const double v = p.samples[(int64_t)s * p.sample_stride + (p.row0 + row) * K + k];
            X[e] = v;
            if constexpr (FAST) {
                Xf[e] = (float)v;
                big = fmaxf(big, fabsf((float)v));
            }
        }
#pragma unroll
        for (int o = 16; o >= 1; o >>= 1) big = fmaxf(big, __shfl_xor_sync(kAll, big, o));
        __syncwarp();
        // Error of an FP32 squared distance d of rounded vectors with entries up to `big` (a mean
        // of samples is no larger): each difference is off by at most eta = 2^-22 big, so d by at
        // most 2 eta sqrt(K d) + K eta^2 + (K + 3) 2^-23 d; twice that is allowed for.
        const float eta = 0x1p-22f * big;
        auto slack = [&](float d) {
            return 2.f * (2.f * eta * sqrtf(K * d) + K * eta * eta + (K + 3) * 0x1p-23f * d) + 1e-36f;
        };
        const float lamf = (float)p.lambda;
        int n = 0;
        bool too_many = false;
        if (p.mode != 0 && S > 0) {
            n = 1;
            for (int k = lane; k < K; k += 32) {
                cen[k] = X[k];
                if constexpr (FAST) cenf[k] = Xf[k];
            }
            for (int i = lane; i < S; i += 32) prev[i] = -1;
            __syncwarp();
            for (int it = 0; it < 100 && !too_many; ++it) {
                const int n0 = n;    // centres at the start of the round: cen; later ones: samples
                auto centre = [&](int c) { return c < n0 ? cen + (size_t)c * K : X + (size_t)opened[c - n0] * K; };
                auto beyond = [&](int i, int c, float d) -> int {   // FP64 distance > lambda
                    if (FAST && fabsf(d - lamf) > slack(d) + 0x1p-22f * lamf) return d > lamf;
                    return sqdist(X + (size_t)i * K, centre(c), K) > p.lambda;
                };
                // nearest existing centre of every sample (lowest index on ties)
                for (int i = lane; i < S; i += 32) {
                    int b = 0;
                    float d1 = INFINITY, d2 = INFINITY;   // smallest and second smallest
                    for (int c = 0; FAST && c < n0; ++c) {
                        const float d = sqdist32(Xf + (size_t)i * K, cenf + (size_t)c * K, K);
                        if (d < d1) {
                            d2 = d1;
                            d1 = d;
                            b = c;
                        } else {
                            d2 = fminf(d2, d);
                        }
                    }
                    // a NaN distance never compares smaller: the FP64 procedure decides
                    if (!FAST || (n0 > 1 && !(d2 - d1 > slack(d1) + slack(d2))) || !(d1 < INFINITY)) {
                        double db = INFINITY;
                        b = 0;
                        for (int c = 0; c < n0; ++c) {
                            const double d = sqdist(X + (size_t)i * K, cen + (size_t)c * K, K);
                            if (d < db) {
                                db = d;
                                b = c;
                            }
                        }
                        d1 = (float)db;
                        far[i] = db > p.lambda;
                    } else {
                        far[i] = beyond(i, b, d1);
                    }
                    assign[i] = b;
                    dbf[i] = d1;
                }
                __syncwarp();
                // samples in order: the next one farther than lambda from every centre opens a
                // cluster; the later samples then compare with the new centre too
                int pos = 0;
                while (pos < S) {
                    int found = S;
                    for (int base = pos; base < S && found == S; base += 32) {
                        const int i = base + lane;
                        const unsigned v = __ballot_sync(kAll, i < S && far[i] != 0);
                        if (v) found = base + __ffs(v) - 1;
                    }
                    if (found == S) break;
                    if (n >= cap) {
                        too_many = true;
                        break;
                    }
                    const int c = n++;
                    if (lane == 0) {
                        opened[c - n0] = found;
                        assign[found] = c;
                    }
                    __syncwarp();
                    for (int j = found + 1 + lane; j < S; j += 32) {
                        float d = 0.f, o = 0.f;
                        if constexpr (FAST) d = sqdist32(Xf + (size_t)j * K, Xf + (size_t)found * K, K), o = dbf[j];
                        bool nearer = d < o;
                        if (!FAST || !(fabsf(d - o) > slack(d) + slack(o)))
                            nearer = sqdist(X + (size_t)j * K, X + (size_t)found * K, K) <
                                     sqdist(X + (size_t)j * K, centre(assign[j]), K);
                        if (nearer) {
                            dbf[j] = d;
                            assign[j] = c;
                            far[j] = beyond(j, c, d);
                        }
                    }
                    __syncwarp();
                    pos = found + 1;
                }
                if (too_many) break;
                for (int c = lane; c < n; c += 32) cnt[c] = 0;
                __syncwarp();
                for (int i = lane; i < S; i += 32) atomicAdd(&cnt[assign[i]], 1);
                __syncwarp();
                // empty clusters are dropped (renumbered in order); offsets of the member lists
                int m = 0;
                for (int c0 = 0; c0 < n; c0 += 32) {
                    const int c = c0 + lane;
                    const unsigned v = __ballot_sync(kAll, c < n && cnt[c] > 0);
                    if (c < n) map[c] = cnt[c] > 0 ? m + __popc(v & ((1u << lane) - 1u)) : -1;
                    m += __popc(v);
                }
                __syncwarp();
                int changed = 0;
                for (int i = lane; i < S; i += 32) {
                    const int a = map[assign[i]];
                    assign[i] = a;
                    changed |= a != prev[i];
                    prev[i] = a;
                }
                __syncwarp();
                // counts move down to their new numbers (a warp of them at a time, in order)
                for (int c0 = 0; c0 < n; c0 += 32) {
                    const int c = c0 + lane;
                    const int to = c < n ? map[c] : -1, v = c < n ? cnt[c] : 0;
                    __syncwarp();
                    if (to >= 0) cnt[to] = v;
                    __syncwarp();
                }
                n = m;
                if (lane == 0) {
                    int s = 0;
                    for (int c = 0; c < n; ++c) off[c] = s, s += cnt[c];
                    off[n] = s;
                }
                __syncwarp();
                for (int c = lane; c < n; c += 32) map[c] = off[c];   // next free place
                __syncwarp();
                for (int i0 = 0; i0 < S; i0 += 32) {
                    const int i = i0 + lane;
                    const int a = i < S ? assign[i] : -1;
                    const unsigned same = __match_any_sync(kAll, a);
                    const int rank = __popc(same & ((1u << lane) - 1u));
                    const int at = a >= 0 ? map[a] : 0;
                    __syncwarp();
                    if (a >= 0) {
                        member[at + rank] = i;
                        if (rank == 0) map[a] = at + __popc(same);
                    }
                    __syncwarp();
                }
                // centres to the means of their samples, in order
                for (int e = lane; e < n * K; e += 32) {
                    const int c = e / K, k = e % K;
                    double s = 0.0;
                    for (int q = off[c]; q < off[c + 1]; ++q) s = dadd(s, X[(size_t)member[q] * K + k]);
                    const double mean = s / (double)cnt[c];
                    cen[e] = mean;
                    if constexpr (FAST) cenf[e] = (float)mean;
                }
                __syncwarp();
                if (!__any_sync(kAll, changed)) break;
            }
        }
        if (too_many) {
            if (lane == 0) over[atomicAdd(over_n, 1)] = (int32_t)row;
            continue;
        }
        if (p.assign)
            for (int i = lane; i < S; i += 32) p.assign[row * S + i] = p.mode != 0 ? assign[i] : 0;
        // the chosen clusters, largest first (ties: lowest index), with at least K + 1 samples
        const int64_t q = p.pi ? row : p.row0 + row;
        int used = 0;
        if (p.mode != 0) {
            const int want = p.mode == 1 ? 1 : C;
            for (int t = 0; t < want; ++t) {
                int best = -1, size = -1;
                for (int c = lane; c < n; c += 32)
                    if (cnt[c] > size) size = cnt[c], best = c;
                // the warp's largest (size, then lowest index) as one key
                unsigned key = best < 0 ? 0u : (unsigned)size << 16 | (0xffffu - (unsigned)best);
                key = __reduce_max_sync(kAll, key);
                if (key == 0u) break;
                best = 0xffff - (int)(key & 0xffffu);
                size = (int)(key >> 16);
                __syncwarp();
                if (lane == 0) cnt[best] = -1;
                __syncwarp();
                if (size < K + 1) break;      // the remaining ones are no larger
                if (lane == 0) map[used] = best;
                ++used;
            }
        }
        __syncwarp();
        // centred members in place, then the packed covariances of all chosen clusters
        for (int t = 0; t < used; ++t) {
            const int c = map[t], b0 = off[c], m = off[c + 1] - b0;
            for (int e = lane; e < m * K; e += 32) {
                const int k = e % K;
                X[(size_t)member[b0 + e / K] * K + k] -= cen[(size_t)c * K + k];
            }
            for (int k = lane; k < K; k += 32) fs.mean(q, t, k) = cen[(size_t)c * K + k];
            if (lane == 0) fs.size(q, t) = (double)m;
        }
        if (lane == 0 && used < C) fs.size(q, used) = 0.0;
        __syncwarp();
        for (int e = lane; e < used * NT; e += 32) {
            const int t = e / NT, c = map[t];
            int i = 0, j = e % NT;
            while (j > i) j -= ++i;
            double s = 0.0;
            for (int b = off[c]; b < off[c + 1]; ++b) {
                const double *x = X + (size_t)member[b] * K;
                s = fma(x[i], x[j], s);
            }
            fs.cov(q, t, e % NT) = s / (double)(off[c + 1] - off[c]);
        }
    }
}

// The rows' precisions from their covariances, one thread per row (FP64 warp instructions cost the
// same whatever their active lanes: a warp per row spent 32 times the instructions, and its
// serial Cholesky and divisions their latency): component precisions (a component with a singular
// covariance is dropped; a row without one takes all its samples), the mixture's pooled mean and
// covariance sum_c pi_c (Sigma_c + (mu_c - m)(mu_c - m)^T), its precision, and the outputs.
__global__ void __launch_bounds__(kRowBlock) fit_kernel(SummaryParams p)
{
    extern __shared__ double sh[];
    const int t = threadIdx.x, rb = blockDim.x;
    const int64_t row = (int64_t)blockIdx.x * rb + t;
    if (row >= p.n_rows) return;
    const int K = p.K, S = p.S, C = p.C, NT = ntri(K);
    const int64_t q = p.pi ? row : p.row0 + row, KK = (int64_t)K * K, W = 1 + 2 * K + NT;
    const FitStage fs = fit_stage(p);
    double *A = sh + t, *Acc = A + NT * rb, *v = Acc + NT * rb, *pm = v + K * rb;
    auto bad_row = [&]() {
        atomicOr(&p.err->flags, ERR_NOT_PD);
        atomicMin(&p.err->first_bad_row, (int)(p.row0 + row));
    };
    // component c's precision (packed in A) to its place
    auto keep_component = [&](int c, double logdet) {
        if (p.pi) {
            for (int i = 0; i < K; ++i)
                for (int j = 0; j <= i; ++j) {
                    const double l = RS(A, tri(i, j));
                    p.Lam[(q * C + c) * KK + i * K + j] = l;
                    p.Lam[(q * C + c) * KK + j * K + i] = l;
                }
        } else if (p.mix) {
            double *o = p.mix + (q * C + c) * W;
            o[0] = logdet;    // + log pi once the weights are known
            for (int e = 0; e < NT; ++e) o[1 + K + e] = RS(A, e);
            for (int i = 0; i < K; ++i) {
                double s = 0.0;
                for (int k = 0; k < K; ++k)
                    s = fma(RS(A, i >= k ? tri(i, k) : tri(k, i)), o[1 + k], s);
                o[1 + K + NT + i] = s;
            }
        }
    };
    double w[kMaxComponents] = {0.0, 0.0, 0.0, 0.0};
    // components whose precision exists add their covariance to the pooled one in Acc
    double tot = 0.0;
    int got = 0;
    for (int e = 0; e < NT; ++e) RS(Acc, e) = 0.0;
    auto add = [&](int src, int dst, double size) -> bool {
        for (int e = 0; e < NT; ++e) RS(A, e) = fs.cov(q, src, e);
        double logdet = 0.0;
        if (!row_spd_inverse(A, v, K, rb, p.mix ? &logdet : nullptr)) return false;
        for (int e = 0; e < NT; ++e) RS(Acc, e) = fma(size, fs.cov(q, src, e), RS(Acc, e));
        if (dst != src)
            for (int k = 0; k < K; ++k) fs.mean(q, dst, k) = fs.mean(q, src, k);
        keep_component(dst, logdet);
        w[dst] = size;
        tot += size;
        return true;
    };
    for (int c = 0; c < C && p.mode != 0; ++c) {
        const double size = fs.size(q, c);
        if (!(size > 0.0)) break;
        if (add(c, got, size)) ++got;
    }
    if (got == 0) {
        // moment matching over all samples
        bool ok = S >= K + 1;
        if (ok) {
            const double *x = p.samples + (p.row0 + row) * K;
            for (int k = 0; k < K; ++k) {
                double s = 0.0;
                for (int i = 0; i < S; ++i) s = dadd(s, x[(int64_t)i * p.sample_stride + k]);
                fs.mean(q, 0, k) = s / (double)S;
            }
            for (int e = 0; e < NT; ++e) RS(A, e) = 0.0;
            for (int i = 0; i < S; ++i) {
                for (int k = 0; k < K; ++k) RS(v, k) = x[(int64_t)i * p.sample_stride + k] - fs.mean(q, 0, k);
                for (int a = 0; a < K; ++a)
                    for (int b = 0; b <= a; ++b) RS(A, tri(a, b)) = fma(RS(v, a), RS(v, b), RS(A, tri(a, b)));
            }
            for (int e = 0; e < NT; ++e) fs.cov(q, 0, e) = RS(A, e) / (double)S;
            ok = add(0, 0, 1.0);
        }
        if (!ok) {
            bad_row();
            return;
        }
        got = 1;
    }
    // pooled mean, and the components' spread about it
    for (int i = 0; i < K; ++i) {
        double s = 0.0;
        for (int c = 0; c < got; ++c) s = fma(w[c] / tot, fs.mean(q, c, i), s);
        RS(pm, i) = s;
    }
    for (int c = 0; c < got; ++c) {
        for (int i = 0; i < K; ++i) RS(v, i) = fs.mean(q, c, i) - RS(pm, i);
        for (int i = 0; i < K; ++i) {
            const double wi = w[c] * RS(v, i);
            for (int j = 0; j <= i; ++j) RS(Acc, tri(i, j)) = fma(wi, RS(v, j), RS(Acc, tri(i, j)));
        }
    }
    const double inv = 1.0 / tot;
    for (int e = 0; e < NT; ++e) RS(A, e) = RS(Acc, e) * inv;
    if (!row_spd_inverse(A, v, K, rb, nullptr)) {
        bad_row();
        return;
    }
    if (p.pi) {
        for (int c = 0; c < C; ++c) {
            p.pi[q * C + c] = c < got ? w[c] / tot : 0.0;
            for (int k = 0; k < K && c >= got; ++k) p.mu[(q * C + c) * K + k] = 0.0;
            for (int64_t e = 0; e < KK && c >= got; ++e) p.Lam[(q * C + c) * KK + e] = 0.0;
        }
        for (int i = 0; i < K; ++i) {
            p.pooled_mu[q * K + i] = RS(pm, i);
            for (int j = 0; j <= i; ++j) {
                p.pooled_Lam[q * KK + i * K + j] = RS(A, tri(i, j));
                p.pooled_Lam[q * KK + j * K + i] = RS(A, tri(i, j));
            }
        }
    }
    if (p.mm_mu) {
        // the summary the library propagates and aggregates: the dominant component (mode 1:
        // one component, so its pooled moments are its own) or the pooled moments, as mean,
        // packed precision and precision x mean
        for (int k = 0; k < K; ++k) p.mm_mu[q * K + k] = RS(pm, k);
        for (int e = 0; e < NT; ++e) p.mm_L[(int64_t)e * p.R + q] = RS(A, e);
        for (int i = 0; i < K; ++i) {
            double s = 0.0;
            for (int k = 0; k < K; ++k) s = fma(RS(A, i >= k ? tri(i, k) : tri(k, i)), RS(pm, k), s);
            p.mm_b[(int64_t)i * p.R + q] = s;
        }
        // mixture store: [log pi + log det(Lambda)/2][mu][L packed][Lambda mu]; unused
        // components get a -infinity score
        for (int c = 0; p.mix && c < C; ++c) {
            double &score = p.mix[(q * C + c) * W];
            score = c < got ? log(w[c] / tot) + score : -INFINITY;
        }
    }
}

cudaError_t launch_summary(const SummaryParams &p, cudaStream_t st)
{
    if (p.n_rows <= 0) return cudaSuccess;
    // first launch: a warp per row with room for kFastCentres clusters; second: the listed rows
    const int cap = kFastCentres, all = 2 * p.S + 1;
    const size_t smem = cluster_smem(p.K, p.S, cap, true), smem_all = cluster_smem(p.K, p.S, all, false);
    cudaError_t e = cudaSuccess;
    // samples too many for the FP32 copies to fit beside them: every row takes the second form
    const bool fast = smem <= 200 * 1024;
    // the second in FP32 distances too where the copies of samples and as many centres fit
    const size_t smem_wide = cluster_smem(p.K, p.S, all, true);
    const bool wide = fast && smem_wide <= kSmemBlock;
    if (fast) e = allow_smem(cluster_kernel<true>, std::max(smem, wide ? smem_wide : 0), kSmemBlock);   // (no static arrays)
    if (e == cudaSuccess) e = allow_smem(cluster_kernel<false>, smem_all, kSmemBlock);
    if (e == cudaSuccess) e = cudaMemsetAsync(p.over_n, 0, sizeof(int32_t), st);
    int dev = 0, sms = 0;
    if (e == cudaSuccess) e = cudaGetDevice(&dev);
    if (e == cudaSuccess) e = cudaDeviceGetAttribute(&sms, cudaDevAttrMultiProcessorCount, dev);
    if (e != cudaSuccess) return e;
    // how many rows are listed is not known here: as many warps as fit on the GPU step through the list.
    // 20,000 rows of 200 samples at K = 10 that all open 200, 60 or 40 clusters: 134.7, 52.2, 38.6 ms with
    // a warp each in FP64; 256, 118, 85 ms with two warps per SM after the first launch; 34, 16, 13 ms now
    auto warps = [&](size_t bytes) {
        return (unsigned)std::min<int64_t>(p.n_rows, (int64_t)sms * std::min<size_t>(32, kSmemBlock / (bytes + 1024) + 1));
    };
    if (fast) {
        cluster_kernel<true><<<(unsigned)p.n_rows, 32, smem, st>>>(p, cap, nullptr, nullptr, p.over, p.over_n);
        if (p.mode != 0 && wide)
            cluster_kernel<true><<<warps(smem_wide), 32, smem_wide, st>>>(p, all, p.over, p.over_n, nullptr, nullptr);
        else if (p.mode != 0)
            cluster_kernel<false><<<warps(smem_all), 32, smem_all, st>>>(p, all, p.over, p.over_n, nullptr, nullptr);
    } else {
        cluster_kernel<false><<<(unsigned)p.n_rows, 32, smem_all, st>>>(p, all, nullptr, nullptr, nullptr, nullptr);
    }
    const size_t per = 2 * (size_t)ntri(p.K) + 2 * p.K;
    const int rb = row_block(per);
    const size_t fit = per * rb * sizeof(double);
    e = allow_smem(fit_kernel, fit);
    if (e != cudaSuccess) return e;
    fit_kernel<<<(unsigned)((p.n_rows + rb - 1) / rb), rb, fit, st>>>(p);
    return cudaGetLastError();
}

// ------------------------------------------------------------------------------------------
// Component choice of a mixture prior: score_c = log pi_c + log det(Lambda_c)/2
// - (x - mu_c)^T Lambda_c (x - mu_c) / 2 at the row's current x (the quadratic form summed in
// order, separate multiplies and adds); the best (lowest index on ties) becomes the prior.
// ------------------------------------------------------------------------------------------
__global__ void mix_choose_kernel(MixChooseParams p)
{
    const int64_t q = (int64_t)blockIdx.x * blockDim.x + threadIdx.x;
    if (q >= p.n) return;
    const int64_t r = p.r0 + q;
    if (!p.has_mix[r]) return;
    const int K = p.K, C = p.C, NT = K * (K + 1) / 2, W = 1 + 2 * K + NT;
    const double *mx = p.mix + r * (int64_t)C * W;
    const double *x = p.X + r * K;
    int bestc = -1;
    double sbest = -INFINITY;
    for (int c = 0; c < C; ++c) {
        const double *o = mx + (int64_t)c * W;
        if (!(o[0] > -INFINITY)) continue;
        const double *m = o + 1, *L = o + 1 + K;
        double qf = 0.0;
        for (int a = 0; a < K; ++a) {
            double s = 0.0;
            for (int b = 0; b < K; ++b)
                s = dadd(s, dmul(L[a >= b ? a * (a + 1) / 2 + b : b * (b + 1) / 2 + a], dsub(x[b], m[b])));
            qf = dadd(qf, dmul(dsub(x[a], m[a]), s));
        }
        const double score = o[0] - 0.5 * qf;
        if (bestc < 0 || score > sbest) {
            bestc = c;
            sbest = score;
        }
    }
    if (bestc < 0) {
        atomicOr(&p.err->flags, ERR_NOT_PD);
        atomicMin(&p.err->first_bad_row, (int)r);
        return;
    }
    const double *o = mx + (int64_t)bestc * W;
    for (int e = 0; e < NT; ++e) p.pL[(int64_t)e * p.R + r] = o[1 + K + e];
    for (int i = 0; i < K; ++i) p.pb[(int64_t)i * p.R + r] = o[1 + K + NT + i];
    if (p.chosen) p.chosen[r] = bestc;
}

void launch_mix_choose(const MixChooseParams &p, cudaStream_t st)
{
    if (p.n <= 0) return;
    mix_choose_kernel<<<(unsigned)((p.n + 127) / 128), 128, 0, st>>>(p);
}

}  // namespace bmf
