// rows.cuh -- thread-per-row FP64 linear algebra on packed lower matrices in interleaved shared
// memory, shared by moment matching and by both entries of Algorithm 2 (misc.cu,
// aggregate_static.cu).
#pragma once
#include "common.cuh"

namespace bmf {

// Entry e of a thread's matrix is at base[e * rb], rb = threads per block (32, fewer when K is large enough
// that 32 rows' matrices would not fit in shared memory).
constexpr int kRowBlock = 32;
constexpr size_t kRowSmemCap = 200 * 1024;
#define RS(base, e) (base)[(e) * rb]

// Threads per block of a thread-per-row kernel holding `per_row` doubles per row.
inline int row_block(size_t per_row)
{
    const size_t fit = kRowSmemCap / (per_row * sizeof(double));
    return (int)(fit >= (size_t)kRowBlock ? kRowBlock : (fit < 1 ? 1 : fit));
}

// In-place packed lower Cholesky (Crout order) with one reciprocal square root per pivot and no
// division: L_jj in P, 1 / L_jj in ri.  Returns false if a pivot is not > 0.
static __device__ bool row_chol(double *P, double *ri, int K, int rb)
{
    for (int j = 0; j < K; ++j) {
        const int jj = tri(j, 0);
        double d = RS(P, jj + j);
        for (int k = 0; k < j; ++k) d = fma(-RS(P, jj + k), RS(P, jj + k), d);
        if (!(d > 0.0)) return false;
        const double rs = rsqrt(d);
        RS(ri, j) = rs;
        RS(P, jj + j) = d * rs;
        for (int i = j + 1; i < K; ++i) {
            const int ii = tri(i, 0);
            double s = RS(P, ii + j);
            for (int k = 0; k < j; ++k) s = fma(-RS(P, ii + k), RS(P, jj + k), s);
            RS(P, ii + j) = s * rs;
        }
    }
    return true;
}

// Solve (L L^T) x = b in place in vector v (interleaved), L packed in P, 1 / L_ii in ri.
static __device__ void row_solve(const double *P, const double *ri, double *v, int K, int rb)
{
    for (int i = 0; i < K; ++i) {
        const int ii = tri(i, 0);
        double s = RS(v, i);
        for (int k = 0; k < i; ++k) s = fma(-RS(P, ii + k), RS(v, k), s);
        RS(v, i) = s * RS(ri, i);
    }
    for (int i = K - 1; i >= 0; --i) {
        double s = RS(v, i);
        for (int k = i + 1; k < K; ++k) s = fma(-RS(P, tri(k, i)), RS(v, k), s);
        RS(v, i) = s * RS(ri, i);
    }
}

// Inverse of the packed SPD matrix A in place; v: K scratch slots.  A = L L^T in place, then
// W = L^{-1} in place (columns left to right; W_ij = -(1/L_ii) sum_{k=j}^{i-1} L_ik W_kj reads only
// entries of L right of column j and entries of W already written), then A^{-1} = W^T W in place
// (rows top to bottom through v: row i needs only rows k >= i of W).  K^3/2 multiply-adds and no
// division.  logdet (nullable): log det(A^{-1}) / 2 = sum log(1 / L_ii).  False if a pivot is not > 0.
static __device__ bool row_spd_inverse(double *A, double *v, int K, int rb, double *logdet)
{
    if (!row_chol(A, v, K, rb)) return false;
    if (logdet) {
        double s = 0.0;
        for (int i = 0; i < K; ++i) s += log(RS(v, i));
        *logdet = s;
    }
    for (int j = 0; j < K; ++j) {
        RS(A, tri(j, j)) = RS(v, j);
        for (int i = j + 1; i < K; ++i) {
            const int ii = tri(i, 0);
            double s = 0.0;
            for (int k = j; k < i; ++k) s = fma(RS(A, ii + k), RS(A, tri(k, j)), s);
            RS(A, ii + j) = -s * RS(v, i);
        }
    }
    for (int i = 0; i < K; ++i) {
        for (int j = 0; j <= i; ++j) {
            double s = 0.0;
            for (int k = i; k < K; ++k) s = fma(RS(A, tri(k, i)), RS(A, tri(k, j)), s);
            RS(v, j) = s;
        }
        for (int j = 0; j <= i; ++j) RS(A, tri(i, j)) = RS(v, j);
    }
    return true;
}

// In-place packed lower Cholesky used only as a positive-definiteness test (pivot > 0 at every
// step), scaling by one reciprocal per column.
static __device__ bool row_pd_test(double *P, int K, int rb)
{
    for (int j = 0; j < K; ++j) {
        const int jj = tri(j, 0);
        double d = RS(P, jj + j);
        for (int k = 0; k < j; ++k) d = fma(-RS(P, jj + k), RS(P, jj + k), d);
        if (!(d > 0.0)) return false;
        const double r = rsqrt(d);
        for (int i = j + 1; i < K; ++i) {
            const int ii = tri(i, 0);
            double s = RS(P, ii + j);
            for (int k = 0; k < j; ++k) s = fma(-RS(P, ii + k), RS(P, jj + k), s);
            RS(P, ii + j) = s * r;
        }
    }
    return true;
}

// Smallest eigenvalue of the symmetric matrix held packed-lower in A (interleaved; destroyed):
// Householder reduction to tridiagonal form T = Q^T A Q (Golub & Van Loan, Algorithm 8.3.1),
// then bisection on the Sturm count of T (the sign changes of the leading principal minors of
// T - x I equal the number of eigenvalues below x; Golub & Van Loan, Section 8.4.1) to an
// interval of 2^-50 |T|, the rounding level of the count.  The result is the smallest
// eigenvalue to O(2^-50 |A|).  v: K scratch slots, dg / of: the K diagonal and K - 1
// off-diagonal entries of T (of: their squares, scaled, after the reduction).
static __device__ double min_eig_tridiag(double *A, double *v, double *dg, double *of, int K, int rb)
{
#define AP(i, j) RS(A, (i) >= (j) ? tri(i, j) : tri(j, i))
    for (int k = 0; k + 2 < K; ++k) {
        // Householder vector of the column below the diagonal, x = A(k+1 .., k)
        double nrm2 = 0.0;
        for (int i = k + 1; i < K; ++i) nrm2 = fma(AP(i, k), AP(i, k), nrm2);
        RS(dg, k) = AP(k, k);
        const double x0 = AP(k + 1, k);
        if (nrm2 == 0.0) {
            RS(of, k) = 0.0;
            continue;
        }
        const double nrm = sqrt(nrm2);
        const double alpha = x0 >= 0.0 ? -nrm : nrm;   // H x = alpha e_1
        RS(of, k) = alpha;
        const double beta = 1.0 / (nrm2 - x0 * alpha);  // 2 / (v^T v), v = x - alpha e_1
        for (int i = k + 1; i < K; ++i) RS(v, i) = AP(i, k);
        RS(v, k + 1) = x0 - alpha;
        // p = beta B v (B the trailing block), then w = p - (beta p^T v / 2) v; the w values
        // replace column k of A, which is not read again
        double pv = 0.0;
        for (int i = k + 1; i < K; ++i) {
            double s = 0.0;
            for (int j = k + 1; j < K; ++j) s = fma(AP(i, j), RS(v, j), s);
            s *= beta;
            RS(A, tri(i, k)) = s;
            pv = fma(s, RS(v, i), pv);
        }
        const double kk = 0.5 * beta * pv;
        for (int i = k + 1; i < K; ++i) RS(A, tri(i, k)) = fma(-kk, RS(v, i), RS(A, tri(i, k)));
        // B -= v w^T + w v^T (lower triangle)
        for (int i = k + 1; i < K; ++i) {
            const double vi = RS(v, i), wi = RS(A, tri(i, k));
            for (int j = k + 1; j <= i; ++j)
                RS(A, tri(i, j)) = fma(-vi, RS(A, tri(j, k)), fma(-wi, RS(v, j), RS(A, tri(i, j))));
        }
    }
    if (K >= 2) {
        RS(dg, K - 2) = AP(K - 2, K - 2);
        RS(of, K - 2) = AP(K - 1, K - 2);
    }
    RS(dg, K - 1) = AP(K - 1, K - 1);
#undef AP
    // Gershgorin interval of T; lambda_min <= min_i T_ii (the Rayleigh quotient of e_i) lowers
    // its top end
    double lo = 0.0, hi = 0.0, dmin = 0.0;
    for (int i = 0; i < K; ++i) {
        const double r = (i > 0 ? fabs(RS(of, i - 1)) : 0.0) + (i + 1 < K ? fabs(RS(of, i)) : 0.0);
        const double a = RS(dg, i) - r, b = RS(dg, i) + r;
        lo = i == 0 ? a : fmin(lo, a);
        hi = i == 0 ? b : fmax(hi, b);
        dmin = i == 0 ? RS(dg, i) : fmin(dmin, RS(dg, i));
    }
    const double nrm = fmax(fabs(lo), fabs(hi));
    if (!(nrm > 0.0)) return 0.0;
    // T / s with s the power of two at or above the norm bound (exact scaling): entries and the
    // bisection interval within [-1, 1], so the Sturm sequence below neither overflows nor, short
    // of K near-coincident eigenvalues, underflows
    const int se = ilogb(nrm) + 1;
    for (int i = 0; i < K; ++i) RS(dg, i) = scalbn(RS(dg, i), -se);
    for (int i = 0; i + 1 < K; ++i) {
        const double e = scalbn(RS(of, i), -se);
        RS(of, i) = e * e;
    }
    lo = scalbn(lo, -se);
    hi = fmin(scalbn(hi, -se), scalbn(dmin, -se) + 0x1.0p-44);
    // bisection on the Sturm count: the number of sign changes of p_0 = 1, p_1 = d_0 - x,
    // p_{i+1} = (d_i - x) p_i - e_{i-1}^2 p_{i-1} (the leading principal minors of T - x I, a zero
    // taking the sign opposite to its predecessor) is the number of eigenvalues below x
    // (Golub & Van Loan, Section 8.4.1); no division, signs read from the bit patterns
    for (int it = 0; it < 100 && hi - lo > 0x1.0p-50; ++it) {
        const double x = 0.5 * (lo + hi);
        double pm = 1.0, pc = RS(dg, 0) - x;
        long long bc = __double_as_longlong(pc);
        unsigned sc = (bc << 1) == 0 ? 1u : (unsigned)((unsigned long long)bc >> 63);
        unsigned below = sc;
        for (int i = 1; i < K; ++i) {
            double pn = fma(RS(dg, i) - x, pc, -RS(of, i - 1) * pm);
            const int em = max((int)((__double_as_longlong(pn) >> 52) & 0x7ff),
                               (int)((__double_as_longlong(pc) >> 52) & 0x7ff));
            if (em < 1023 - 600) {
                // both terms below 2^-600: rescale them by the same power of two (exact)
                const double f = scalbn(1.0, 1023 - max(em, 1));
                pn *= f;
                pc *= f;
            }
            const long long b2 = __double_as_longlong(pn);
            const unsigned sn = (b2 << 1) == 0 ? (sc ^ 1u) : (unsigned)((unsigned long long)b2 >> 63);
            below += sn ^ sc;
            pm = pc;
            pc = pn;
            sc = sn;
        }
        if (below >= 1)
            hi = x;
        else
            lo = x;
    }
    return scalbn(0.5 * (lo + hi), se);
}

// Threads per block for a thread-per-row kernel with `per_row` shared slots: at most
// kRowBlock, fewer when the block would not leave room for four blocks per SM.
inline int row_block_small(size_t per_row)
{
    const size_t fit = (size_t)(220 * 1024 / 4) / (per_row * sizeof(double));
    return (int)(fit >= (size_t)kRowBlock ? kRowBlock : (fit < 1 ? 1 : fit));
}

}  // namespace bmf
