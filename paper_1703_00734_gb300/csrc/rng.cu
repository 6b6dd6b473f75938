// rng.cu -- the device generator of the Gibbs sweep's random numbers.
//
// Counter-based: Philox4x64-10 (Salmon, Moraes, Dror, Shaw, "Parallel random numbers: as easy
// as 1, 2, 3", SC'11) with key (seed, 0) and counter (index, t, tag, attempt), t the 1-based
// sweep number of the subset's chain and tag = subset id * 256 + factor * 16 + kind.  Every
// number is a pure function of its position, so the draws do not depend on batching, on the
// launch shape, on the precision mode or on how sweeps are split across calls.  (Their last bits
// depend on the form of the normals, which K alone chooses: tables up to K = 48, the FP64
// functions above.)
//   kind 2 (hyperparameter normals) and kind 3 (z of the rows): element e of the stream comes
//     from call e / 4; words (0, 1) give elements 4q, 4q + 1 and words (2, 3) elements
//     4q + 2, 4q + 3 by Box-Muller (cosine, sine), u1 = (top 53 bits + 1) 2^-53 in (0, 1] and
//     u2 = top 53 bits 2^-53 in [0, 1);
//   kind 1 (chi-square, dof nu0 + n - k for diagonal entry k): 2 Gamma(dof / 2) by Marsaglia &
//     Tsang (ACM TOMS 2000), attempt j on counter (k, t, tag, j): a candidate from the
//     cosine normal of words (0, 1), the acceptance uniform from word 2 and, for shape < 1,
//     the U^(1/a) boost from word 3.  64 rejections in a row set an error flag;
//   kind 4 (chi-square of a sampled noise precision, factor W): variate k drawn the same way
//     with dof 2 a0 + the entries of column k of the subset (one precision per column) or
//     2 a0 + the subset's entries (one precision per subset, k = 0).
// One thread per Philox call (normal streams) or per variate (chi-square).
#include "common.cuh"
#include "fpair.cuh"
#include "kernels.h"

namespace bmf {

__device__ __forceinline__ void philox4x64_10(uint64_t x[4], uint64_t k0, uint64_t k1)
{
    const uint64_t M0 = 0xD2E7470EE14C6C93ull, M1 = 0xCA5A826395121157ull;
#pragma unroll
    for (int r = 0; r < 10; ++r) {
        const uint64_t hi0 = __umul64hi(M0, x[0]), lo0 = M0 * x[0];
        const uint64_t hi1 = __umul64hi(M1, x[2]), lo1 = M1 * x[2];
        const uint64_t n0 = hi1 ^ x[1] ^ k0, n2 = hi0 ^ x[3] ^ k1;
        x[0] = n0;
        x[1] = lo1;
        x[2] = n2;
        x[3] = lo0;
        k0 += 0x9E3779B97F4A7C15ull;
        k1 += 0xBB67AE8584CAA73Bull;
    }
}

__device__ __forceinline__ double u_open0(uint64_t w) { return (double)((w >> 11) + 1) * 0x1.0p-53; }

// Box-Muller on words a and b: r cos(2 pi u2) and r sin(2 pi u2), r = sqrt(-2 ln u1).
//
// The FP64 pipe takes a warp instruction every 17 clocks per SM, and log, sqrt and sincos in FP64
// spend about 100 of them on a pair of normals; the sweeps' own kernels wait beside this one for the
// same pipe.  Here FP64 does only what must carry 53 bits, 16 instructions a pair: the leading
// terms come from tables (Tang 1990's scheme for log; the angle sum for sine and cosine), and
// what is added to them, at most 2^-9 of the result, is taken in float pairs (48 bits).
// 6.4 million normals: 450 us with the FP64 functions, 137 us with this; 2-norm error of the
// normals against long double 2.4e-16 before, 0.94e-16 now (largest error 2.9e-15, now 1.2e-15).

// ln u1 for u1 = U 2^-53, 1 <= U <= 2^53: with U = m 2^k, m in [1, 2), and c the table's
// reciprocal of m's interval, r = m c - 1 (one rounding), |r| < 2^-10:
//   ln u1 = e ln 2 - ln c + r + r^2 (-1/2 + r (1/3 + r (-1/4 + r / 5 - r^2 / 6))).
// From m = 1 + 424/1024 (about sqrt 2) on the table counts m / 2 and e one higher, and the first
// and last interval have c = 1 and 1/2 exactly, so that ln u1 keeps its relative accuracy at 1.
__device__ __forceinline__ double log_unit(uint64_t U, const GenTables *tab)
{
    const int k = 63 - __clzll((long long)U);
    const uint64_t frac = (U << (63 - k)) << 1;              // bits below the leading one
    const int idx = (int)(frac >> 54);
    const double m = __longlong_as_double((long long)(0x3ff0000000000000ull | frac >> 12));
    const double2 t = __ldg(reinterpret_cast<const double2 *>(&tab->lg[idx]));                  // c, -ln c (- ln 2)
    const double r = fma(m, t.x, -1.0);
    const fpair R = split(r);
    const float x = R.h;
    float s, e;
    two_sum(0x1.555556p-2f, x * fmaf(x, fmaf(x, -1.f / 6.f, 0.2f), -0.25f), s, e);
    fpair q = pmul(renorm(s, e - 0x1.555556p-27f), R);       // 1/3 = h + l with l = -2^-25 h
    q = pmul(pmul(R, R), padd(fpair{-0.5f, 0.f}, q));
    const double base = fma((double)(k - 53 + (idx >= kLogHalf ? 1 : 0)), 0.6931471805599453, t.y);
    return base + (r + join(q));
}

// sqrt(t) for t zero or in [2^-53, 2^7]: the FP32 reciprocal square root, then two steps of
// s += (t - s^2) y / 2.
__device__ __forceinline__ double sqrt_unit(double t)
{
    const int hi = __double2hiint(t);
    const float f = __uint_as_float(((unsigned)hi << 3 | (unsigned)__double2loint(t) >> 29) - (896u << 23));
    const double y = widen(rsqrtf(f));
    const double y2 = __hiloint2double(__double2hiint(y) - (1 << 20), __double2loint(y));
    double s = t * y;
    s = fma(fma(-s, s, t), y2, s);
    s = fma(fma(-s, s, t), y2, s);
    return hi == 0 ? 0.0 : s;
}

// The same with the FP64 functions (rounded differently in the last bits), for K > 48.
__device__ __forceinline__ void box_muller_fp64(uint64_t a, uint64_t b, double &z0, double &z1)
{
    const double r = sqrt(-2.0 * log(u_open0(a)));
    double s, c;
    sincos(6.283185307179586 * ((double)(b >> 11) * 0x1.0p-53), &s, &c);
    z0 = r * c;
    z1 = r * s;
}

template <bool TABLES>
__device__ __forceinline__ void box_muller(uint64_t a, uint64_t b, const GenTables *tab, double &z0, double &z1)
{
    if constexpr (!TABLES) {
        box_muller_fp64(a, b, z0, z1);
        return;
    }
    const double ln = log_unit((a >> 11) + 1, tab);
    // -2 ln u1 >= 0 (zero only for u1 = 1)
    const int lh = __double2hiint(ln) & 0x7fffffff;
    const double rad = sqrt_unit(__hiloint2double(lh == 0 ? 0 : lh + (1 << 20), __double2loint(ln)));
    // the angle: N 2^-53 turns = k / 2048 + d 2^-53, |d| <= 2^41
    const int64_t N = (int64_t)(b >> 11);
    const int k = (int)((N + (1ll << 41)) >> 42);
    const int64_t d = N - ((int64_t)k << 42);
    const fpair th = pmul(renorm((float)(int)(d >> 18) * 0x1p18f, (float)(int)(d & 0x3ffff)),
                          fpair{0x1.921fb6p-51f, -0x1.777a5cp-76f});      // 2 pi 2^-53
    const fpair x2 = pmul(th, th);
    // sin th and cos th - 1: what follows their leading terms is below 2^-30 and 2^-42
    const fpair sn = renorm(th.h, fmaf(th.h * x2.h, fmaf(x2.h, 1.f / 120.f, -1.f / 6.f), th.l));
    const fpair cm = renorm(-0.5f * x2.h, fmaf(x2.h * x2.h, 1.f / 24.f, -0.5f * x2.l));
    const SinCos *e = &tab->sc[k & 511];
    const double2 SC = __ldg(reinterpret_cast<const double2 *>(&e->s));
    const float4 p = __ldg(reinterpret_cast<const float4 *>(&e->sp));
    const fpair S{p.x, p.y}, C{p.z, p.w};
    const double c = SC.y + join(renorm(pfnma(pmul(C, cm), S, sn)));
    const double s = SC.x + join(renorm(pfnma(pmul(S, cm), C, fpair{-sn.h, -sn.l})));
    // quadrant: (c, s), (-s, c), (-c, -s), (s, -c)
    const int quad = (k >> 9) & 3;
    const double u = (quad & 1) ? s : c, v = (quad & 1) ? c : s;
    const int nu = (quad == 1 || quad == 2) ? (int)0x80000000 : 0, nv = (quad >= 2) ? (int)0x80000000 : 0;
    z0 = rad * __hiloint2double(__double2hiint(u) ^ nu, __double2loint(u));
    z1 = rad * __hiloint2double(__double2hiint(v) ^ nv, __double2loint(v));
}

template <bool TABLES>
__global__ void __launch_bounds__(256) gen_kernel(GenParams p)
{
    const int64_t u = (int64_t)blockIdx.x * blockDim.x + threadIdx.x;
    if (u >= p.n_units) return;
    int lo = 0, hi = p.n_segs - 1;           // last segment with unit0 <= u
    while (lo < hi) {
        const int mid = (lo + hi + 1) >> 1;
        if (p.segs[mid].unit0 <= u) lo = mid; else hi = mid - 1;
    }
    const GenSeg sg = p.segs[lo];
    const int64_t l = u - sg.unit0;
    double *out = p.out + sg.out;
    if (sg.kind == 1 || sg.kind == 4) {
        // kind 1: the Bartlett diagonal, dof0 - k; kind 4: the noise precision of a column
        // (dof0 + its entries) or of a subset (dof0)
        const double dof = sg.kind == 1 ? sg.dof0 - (double)l
                                        : sg.dof0 + (sg.row0 >= 0
                                                         ? (double)(p.cnt_ptr[sg.row0 + l + 1] -
                                                                    p.cnt_ptr[sg.row0 + l])
                                                         : 0.0);
        const double a = 0.5 * dof;
        const bool boost = a < 1.0;
        const double d = (boost ? a + 1.0 : a) - 1.0 / 3.0, c = 1.0 / sqrt(9.0 * d);
        double res = __longlong_as_double(0x7ff8000000000000ll);
        bool ok = false;
        for (int j = 0; j < 64 && dof > 0.0; ++j) {
            uint64_t w[4] = {(uint64_t)l, (uint64_t)p.t, sg.tag, (uint64_t)j};
            philox4x64_10(w, p.seed, 0);
            double x, unused;
            box_muller<TABLES>(w[0], w[1], p.tab, x, unused);
            double v = 1.0 + c * x;
            if (!(v > 0.0)) continue;
            v = v * v * v;
            const double uu = u_open0(w[2]);
            if (uu < 1.0 - 0.0331 * (x * x) * (x * x) ||
                log(uu) < 0.5 * x * x + d * (1.0 - v + log(v))) {
                double g = d * v;
                if (boost) g *= pow(u_open0(w[3]), 1.0 / a);
                res = 2.0 * g;
                ok = true;
                break;
            }
        }
        if (!ok) atomicOr(&p.err->flags, ERR_RNG);
        out[l] = res;
        return;
    }
    uint64_t w[4] = {(uint64_t)l, (uint64_t)p.t, sg.tag, 0};
    philox4x64_10(w, p.seed, 0);
    double z[4];
    box_muller<TABLES>(w[0], w[1], p.tab, z[0], z[1]);
    box_muller<TABLES>(w[2], w[3], p.tab, z[2], z[3]);
    const int64_t e0 = 4 * l;
#pragma unroll
    for (int q = 0; q < 4; ++q)
        if (e0 + q < sg.count) out[e0 + q] = z[q];
}

void launch_gen(const GenParams &p, cudaStream_t st)
{
    if (p.n_units <= 0) return;
    const unsigned grid = (unsigned)((p.n_units + 255) / 256);
    if (p.tab)
        gen_kernel<true><<<grid, 256, 0, st>>>(p);
    else
        gen_kernel<false><<<grid, 256, 0, st>>>(p);
}

// Host side: the segments of one sweep's draw buffer for a batch (layout of the public header).
int64_t gen_segments(const std::vector<GenSubset> &subs, int K, double nu0, int noise, double a0,
                     std::vector<GenSeg> &segs)
{
    segs.clear();
    const int64_t HN = (int64_t)K * (K - 1) / 2 + K;
    int64_t unit = 0, off = 0;
    auto add = [&](int kind, int64_t count, uint64_t tag, double dof0, int64_t row0 = -1) {
        if (count <= 0) return;
        GenSeg s;
        s.unit0 = unit;
        s.count = count;
        s.out = off;
        s.tag = tag;
        s.dof0 = dof0;
        s.kind = kind;
        s.row0 = row0;
        segs.push_back(s);
        unit += (kind == 1 || kind == 4) ? count : (count + 3) / 4;
        off += count;
    };
    auto tag = [](int sid, int f, int kind) {
        return ((uint64_t)(uint32_t)sid << 8) | ((uint64_t)f << 4) | (uint64_t)kind;
    };
    for (const GenSubset &s : subs)
        for (int f = 0; f < 2; ++f) {
            const int64_t m = f == 0 ? s.n : s.d;
            add(1, K, tag(s.sid, f, 1), nu0 + (double)m);
            add(2, HN, tag(s.sid, f, 2), 0.0);
        }
    for (int f = 0; f < 2; ++f)
        for (const GenSubset &s : subs) add(3, (f == 0 ? s.n : s.d) * K, tag(s.sid, f, 3), 0.0);
    // noise precisions: one chi-square per column (dof 2 a0 + the column's entries) or one per
    // subset (dof 2 a0 + its entries), stream (subset, W, kind 4)
    if (noise == 2)
        for (const GenSubset &s : subs) add(4, s.d, tag(s.sid, 1, 4), 2.0 * a0, s.woff);
    else if (noise == 1)
        for (const GenSubset &s : subs) add(4, 1, tag(s.sid, 1, 4), 2.0 * a0 + (double)s.nnz, -1);
    return unit;
}

}  // namespace bmf
