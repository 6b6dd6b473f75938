// aggregate_static.cu -- bmf_aggregate_static: the aggregation of per-row Gaussian submodels
// (Eq. 14 with the eigenvalue correction of Algorithm 2) for callers that cannot allocate GPU
// memory, e.g. a runtime that owns all device memory through its own allocator and forbids
// libraries from calling cudaMalloc, or a service whose device footprint is fixed at start-up.
//
// What passes between the call's kernels lives in one file-scope static device array of fixed size
// (kStaticBytes).  Every GPU that loads this library holds that array until the process exits.
// All calls share it: the array keeps the previous call's contents, the call clears the part
// that must start at zero, and two calls whose work overlaps on the GPU (different streams or
// different host threads) race on it.  The call reads its counters back and synchronises its
// stream before returning.
#include <algorithm>
#include <cstdint>
#include <mutex>

#include "bmf.h"
#include "common.cuh"
#include "rows.cuh"

namespace bmf {
void set_noctx_error(const char *m);  // message for bmf_last_error(NULL); no allocation
}

namespace {

constexpr size_t kStaticBytes = size_t(32) << 20;                // 32 MiB
constexpr size_t kHeaderDoubles = 32;                             // 256 bytes: counters, flags
constexpr size_t kStaticDoubles = kStaticBytes / sizeof(double);
static_assert(kStaticDoubles - kHeaderDoubles == BMF_AGGREGATE_STATIC_MAX_DOUBLES,
              "public limit and static array disagree");
constexpr int kMaxDevices = 64;

// [0]: number of corrected (row, submodel) pairs (as unsigned long long bits)
// [1]: error flags (bit 0: an aggregated precision is not positive definite)
// [2]: length of the current round's list (as unsigned)
// [kHeaderDoubles ...]: row sums, corrections and list of the current round
static __device__ __align__(256) double g_scratch[kStaticDoubles];

// Submodel Gaussians of the call's rows: mu [J][R][K], Lam [J][R][K][K] (full symmetric).
struct Models {
    int K;
    int64_t R;
    const double *mu, *Lam;
    __device__ const double *L(int64_t j, int64_t n) const { return Lam + (j * R + n) * K * K; }
    __device__ const double *m(int64_t j, int64_t n) const { return mu + (j * R + n) * K; }
};

// The rows [n0, n0 + nr) and submodels [j0, j0 + nj) (j0 >= 1) of one round; pair q of the round
// is row n0 + q % nr with submodel j0 + q / nr.
struct Round {
    int64_t n0, nr;
    int64_t j0, nj;
    bool first, last;            // of the row range's submodel ranges
    double *corr;                // [nj * nr] eigenvalue correction of each pair, 0 for none
    int32_t *list;               // [nj * nr] pairs whose difference is not positive definite
    double *acc;                 // [nr * (ntri(K) + K)] sums between submodel ranges
    unsigned long long *ncorr, *flags;
    unsigned *list_n;
};

__device__ void load_difference(const Models &a, int64_t j, int64_t n, double *F, int rb)
{
    const double *Lj = a.L(j, n), *L1 = a.L(0, n);
    for (int i = 0; i < a.K; ++i)
        for (int k = 0; k <= i; ++k) RS(F, bmf::tri(i, k)) = Lj[i * a.K + k] - L1[i * a.K + k];
}

// The passes of the context's aggregation (misc.cu) on these arrays: a positive-definiteness
// test of every (row, submodel) pair that lists the others, the smallest eigenvalue of the
// listed pairs, then the sums and the solve per row.  All three are bound by the FP64 pipe (a
// warp instruction occupies its scheduler's share for about 64 clocks); splitting them keeps a
// warp's pairs alike and a pair's matrix in shared memory.  A call on 40,000 rows x 4 submodels at
// K = 10: 1.33 ms, against 113 ms for one thread per row running Jacobi rotations in global memory.
__global__ void __launch_bounds__(bmf::kRowBlock) static_pd_kernel(Models a, Round w)
{
    extern __shared__ double sm[];
    const int t = threadIdx.x, rb = blockDim.x;
    const int64_t q = (int64_t)blockIdx.x * rb + t;
    bool listed = false;
    if (q < w.nr * w.nj) {
        load_difference(a, w.j0 + q / w.nr, w.n0 + q % w.nr, sm + t, rb);
        listed = !bmf::row_pd_test(sm + t, a.K, rb);
        if (!listed) w.corr[q] = 0.0;
    }
    const unsigned am = __activemask();
    const unsigned votes = __ballot_sync(am, listed);
    const int lane = t & 31, leader = __ffs(am) - 1;
    unsigned base = 0;
    if (lane == leader && votes) base = atomicAdd(w.list_n, (unsigned)__popc(votes));
    base = __shfl_sync(am, base, leader);
    if (listed) w.list[base + __popc(votes & ((1u << lane) - 1u))] = (int32_t)q;
}

__global__ void __launch_bounds__(bmf::kRowBlock) static_eig_kernel(Models a, Round w, double eps_rel)
{
    extern __shared__ double sm[];
    const int t = threadIdx.x, rb = blockDim.x;
    const int64_t k = (int64_t)blockIdx.x * rb + t, n_list = *w.list_n;
    if (k >= n_list) return;
    if (k == 0) atomicAdd(w.ncorr, (unsigned long long)n_list);
    const int K = a.K;
    const int64_t q = w.list[k], n = w.n0 + q % w.nr;
    const double *L1 = a.L(0, n);
    double mean_diag = 0.0;
    for (int i = 0; i < K; ++i) mean_diag += L1[i * K + i];
    mean_diag /= (double)K;
    const double eps = eps_rel * (mean_diag > 1.0 ? mean_diag : 1.0);
    double *F = sm + t, *v = F + bmf::ntri(K) * rb, *dg = v + K * rb, *of = dg + K * rb;
    load_difference(a, w.j0 + q / w.nr, n, F, rb);
    w.corr[q] = fabs(bmf::min_eig_tridiag(F, v, dg, of, K, rb)) + eps;
}

__global__ void __launch_bounds__(bmf::kRowBlock) static_solve_kernel(Models a, Round w, int64_t J,
                                                                      double *__restrict__ out)
{
    extern __shared__ double sm[];
    const int t = threadIdx.x, rb = blockDim.x;
    const int64_t p = (int64_t)blockIdx.x * rb + t, n = w.n0 + p;
    if (p >= w.nr) return;
    const int K = a.K, NT = bmf::ntri(K);
    double *Ls = sm + t, *h = Ls + NT * rb, *ri = h + K * rb;
    const double *L1 = a.L(0, n);
    if (w.first) {
        const double c0 = 2.0 - (double)J;
        const double *m1 = a.m(0, n);
        for (int i = 0; i < K; ++i) {
            double s = 0.0;
            for (int k = 0; k < K; ++k) s = fma(L1[i * K + k], m1[k], s);
            RS(h, i) = c0 * s;
            for (int k = 0; k <= i; ++k) RS(Ls, bmf::tri(i, k)) = c0 * L1[i * K + k];
        }
    } else {
        for (int e = 0; e < NT + K; ++e) RS(Ls, e) = w.acc[(int64_t)e * w.nr + p];
    }
    for (int64_t jj = 0; jj < w.nj; ++jj) {
        const double *Lj = a.L(w.j0 + jj, n), *mj = a.m(w.j0 + jj, n);
        const double corr = w.corr[jj * w.nr + p];
        // a corrected submodel is (Lambda^(j) - Lambda^(1) + corr I) + Lambda^(1); the lower
        // triangle stands for both, as in the packed form
        auto entry = [&](int i, int k) {
            const int e = i >= k ? i * K + k : k * K + i;
            if (!(corr > 0.0)) return Lj[e];
            double d = Lj[e] - L1[e];
            if (i == k) d += corr;
            return d + L1[e];
        };
        for (int i = 0; i < K; ++i) {
            double s = 0.0;
            for (int k = 0; k < K; ++k) {
                const double l = entry(i, k);
                s = fma(l, mj[k], s);
                if (k <= i) RS(Ls, bmf::tri(i, k)) += l;
            }
            RS(h, i) += s;
        }
    }
    if (!w.last) {
        for (int e = 0; e < NT + K; ++e) w.acc[(int64_t)e * w.nr + p] = RS(Ls, e);
        return;
    }
    if (!bmf::row_chol(Ls, ri, K, rb)) {
        atomicOr(w.flags, 1ull);
        return;
    }
    bmf::row_solve(Ls, ri, h, K, rb);
    for (int i = 0; i < K; ++i) out[n * K + i] = RS(h, i);
}

// Launches of one call: rounds of rows, and of submodels where one row's pairs would not fit in
// the static array (per round: a correction and a list entry per pair, a row's sums).
cudaError_t launch_rounds(int K, int64_t R, int64_t J, const double *mu, const double *Lam,
                          double eps_rel, double *out, double *scr, cudaStream_t st)
{
    const Models a{K, R, mu, Lam};
    const int64_t cap = (int64_t)(kStaticDoubles - kHeaderDoubles), per_row = bmf::ntri(K) + K;
    // a pair takes a correction (one double) and a list entry (half a double)
    const int64_t nj = std::max<int64_t>(1, std::min<int64_t>(J - 1, (cap - per_row) / 2));
    const int64_t nr = std::max<int64_t>(1, std::min<int64_t>(R, cap / (2 * nj + per_row)));
    auto blocks = [](size_t slots, int &rb, size_t &smem) {
        rb = bmf::row_block_small(slots);
        smem = slots * rb * sizeof(double);
    };
    int rp, re, rs;
    size_t sp, se, ss;
    blocks(bmf::ntri(K), rp, sp);
    blocks(bmf::ntri(K) + 3 * K, re, se);
    blocks(bmf::ntri(K) + 2 * K, rs, ss);
    cudaError_t e = cudaSuccess;
    e = bmf::allow_smem(static_pd_kernel, sp);
    if (!e) e = bmf::allow_smem(static_eig_kernel, se);
    if (!e) e = bmf::allow_smem(static_solve_kernel, ss);
    if (e) return e;
    Round w;
    w.ncorr = reinterpret_cast<unsigned long long *>(scr);
    w.flags = reinterpret_cast<unsigned long long *>(scr + 1);
    w.list_n = reinterpret_cast<unsigned *>(scr + 2);
    w.acc = scr + kHeaderDoubles;
    for (w.n0 = 0; w.n0 < R; w.n0 += nr) {
        w.nr = std::min(nr, R - w.n0);
        w.corr = w.acc + w.nr * per_row;
        w.j0 = 1;
        do {
            w.nj = std::min(nj, J - w.j0);
            w.first = w.j0 == 1;
            w.last = w.j0 + w.nj >= J;
            const int64_t pairs = w.nr * w.nj;
            w.list = reinterpret_cast<int32_t *>(w.corr + pairs);
            if (pairs > 0) {
                if ((e = cudaMemsetAsync(w.list_n, 0, sizeof(unsigned), st))) return e;
                static_pd_kernel<<<(unsigned)((pairs + rp - 1) / rp), rp, sp, st>>>(a, w);
                static_eig_kernel<<<(unsigned)((pairs + re - 1) / re), re, se, st>>>(a, w, eps_rel);
            }
            static_solve_kernel<<<(unsigned)((w.nr + rs - 1) / rs), rs, ss, st>>>(a, w, J, out);
            if ((e = cudaGetLastError())) return e;
            w.j0 += w.nj;
        } while (w.j0 < J);
    }
    return cudaSuccess;
}

// Device address of the static array, looked up once per device with that device current and
// kept for the life of the process (a cudaDeviceReset of that device is not supported after it).
std::mutex g_mutex;
double *g_addr[kMaxDevices] = {nullptr};

bool scratch_address(int dev, double **out)
{
    std::lock_guard<std::mutex> lock(g_mutex);
    if (!g_addr[dev]) {
        void *p = nullptr;
        if (cudaGetSymbolAddress(&p, g_scratch) != cudaSuccess || !p) return false;
        g_addr[dev] = static_cast<double *>(p);
    }
    *out = g_addr[dev];
    return true;
}

bmf_status fail(bmf_status s, const char *m)
{
    bmf::set_noctx_error(m);
    return s;
}

}  // namespace

extern "C" bmf_status bmf_aggregate_static(int32_t K, int64_t R, int32_t J, const double *mu,
                                           const double *Lam, double eps_rel, double *mu_star,
                                           int64_t *n_corrected, void *stream)
{
    bmf::set_noctx_error("");
    if (K < 1 || K > 16 || J < 1 || R < 0)
        return fail(BMF_E_ARG, "bmf_aggregate_static: need 1 <= K <= 16, J >= 1, R >= 0");
    if ((uint64_t)R * (uint64_t)K * (uint64_t)K > kStaticDoubles - kHeaderDoubles)
        return fail(BMF_E_SHAPE, "bmf_aggregate_static: R * K * K exceeds the static scratch "
                                 "(BMF_AGGREGATE_STATIC_MAX_DOUBLES); split the rows over calls");
    if (R > 0 && (!mu || !Lam || !mu_star)) return fail(BMF_E_ARG, "bmf_aggregate_static: null pointer");
    int dev = 0;
    if (cudaGetDevice(&dev) != cudaSuccess || dev < 0 || dev >= kMaxDevices)
        return fail(BMF_E_CUDA, "bmf_aggregate_static: no current CUDA device");
    double *scr = nullptr;
    if (!scratch_address(dev, &scr))
        return fail(BMF_E_CUDA, "bmf_aggregate_static: cudaGetSymbolAddress failed");
    cudaStream_t st = static_cast<cudaStream_t>(stream);
    if (cudaMemsetAsync(scr, 0, kHeaderDoubles * sizeof(double), st) != cudaSuccess)
        return fail(BMF_E_CUDA, "bmf_aggregate_static: clearing the counters failed");
    if (R > 0) {
        if (launch_rounds(K, R, J, mu, Lam, eps_rel > 0 ? eps_rel : 1e-6, mu_star, scr, st) != cudaSuccess)
            return fail(BMF_E_CUDA, "bmf_aggregate_static: kernel launch failed");
    }
    unsigned long long head[2] = {0, 0};
    if (cudaMemcpyAsync(head, scr, sizeof(head), cudaMemcpyDeviceToHost, st) != cudaSuccess ||
        cudaStreamSynchronize(st) != cudaSuccess)
        return fail(BMF_E_CUDA, "bmf_aggregate_static: CUDA error");
    if (n_corrected) *n_corrected = (int64_t)head[0];
    if (head[1] & 1ull)
        return fail(BMF_E_NOT_PD, "bmf_aggregate_static: an aggregated precision is not positive definite");
    return BMF_OK;
}
