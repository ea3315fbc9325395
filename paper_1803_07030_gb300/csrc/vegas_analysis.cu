// Analysis of a simulation history on the GPU: thermal averages with binned and jackknife
// errors, the Binder cumulant and the cumulants V1, V2, integrated autocorrelation times
// (Sec. II, Sec. IV.A-B), and single/multiple histogram reweighting (Sec. IV.E; Ferrenberg
// & Swendsen 1988, 1989). FP64 throughout; every sum is a fixed-order block reduction, so
// results do not change between runs.
#include <cuda_runtime.h>

#include <cmath>
#include <cstdint>
#include <cstring>
#include <string>
#include <vector>

#include "vegas_exp64.cuh"
#include "vegas_internal.h"

using namespace vegas;

namespace {

constexpr int kAnaThreads = 256;
constexpr int kMaxObs = 8;  // observables per reweighting call
constexpr int kMultiBatch = 16;  // fused reweighting iterations per host synchronisation

thread_local std::string g_ana_err;

vegas_status ana_fail(vegas_status st, const std::string &m) {
    g_ana_err = m;
    return st;
}

// A host exception caught at an entry point, as a status (called inside a catch block).
vegas_status analysis_host_exception() {
    std::string m;
    const vegas_status st = status_of_current_exception(m);
    return ana_fail(st, m);
}

// Sum of v over the block, in a fixed order; every thread gets the result.
__device__ double block_sum(double v, double *sm) {
    for (int off = 16; off > 0; off >>= 1) v += __shfl_xor_sync(0xFFFFFFFFu, v, off);
    const int lane = threadIdx.x & 31, warp = threadIdx.x >> 5;
    __syncthreads();  // sm may still be read by the previous call
    if (lane == 0) sm[warp] = v;
    __syncthreads();
    double s = 0.0;
    for (int w = 0; w < (int)(blockDim.x >> 5); ++w) s += sm[w];
    return s;
}

// Sums over records [i0, i1) of one series: the eight shifted moments
//   e' = E - Eref, a' = |M| - Aref:  e', e'^2, a', a'^2, a' e', M^2, M^4, M^2 e'.
__device__ void moment_sums(const double *h, int64_t i0, int64_t i1, double Eref, double Aref, double *sm,
                            double out[8]) {
    double v[8] = {0.0, 0.0, 0.0, 0.0, 0.0, 0.0, 0.0, 0.0};
    for (int64_t i = i0 + threadIdx.x; i < i1; i += blockDim.x) {
        const double *r = h + i * 4;
        const double m2 = r[1] * r[1] + r[2] * r[2] + r[3] * r[3];
        const double e = r[0] - Eref, a = sqrt(m2) - Aref;
        v[0] += e;
        v[1] += e * e;
        v[2] += a;
        v[3] += a * a;
        v[4] += a * e;
        v[5] += m2;
        v[6] += m2 * m2;
        v[7] += m2 * e;
    }
    for (int q = 0; q < 8; ++q) out[q] = block_sum(v[q], sm);
}

// (c, chi, u4) from moment sums over n samples.
__device__ void estimates(const double S[8], double n, double N, double T, double out[3]) {
    const double me = S[0] / n, ma = S[2] / n, m2 = S[5] / n;
    out[0] = (S[1] / n - me * me) / (N * T * T);
    out[1] = (S[3] / n - ma * ma) / (N * T);
    out[2] = 1.0 - (S[6] / n) / (3.0 * m2 * m2);
}

// Integrated autocorrelation time of x_i = (E or |M|) - mean, Sokal's window (c = 6).
__device__ double tau_window(const double *h, int64_t cut, int64_t n, int which, double mean, double *sm) {
    auto x = [&](int64_t i) {
        const double *r = h + (cut + i) * 4;
        return (which == 0 ? r[0] : sqrt(r[1] * r[1] + r[2] * r[2] + r[3] * r[3])) - mean;
    };
    double c0 = 0.0;
    for (int64_t i = threadIdx.x; i < n; i += blockDim.x) {
        const double d = x(i);
        c0 += d * d;
    }
    c0 = block_sum(c0, sm) / (double)n;
    if (c0 == 0.0) return 0.5;
    double tau = 0.5;
    for (int64_t t = 1; t <= n / 2; ++t) {
        double c = 0.0;
        for (int64_t i = threadIdx.x; i < n - t; i += blockDim.x) c += x(i) * x(i + t);
        c = block_sum(c, sm) / (double)(n - t);
        tau += c / c0;
        if ((double)t >= 6.0 * tau) break;
    }
    return tau;
}

// One block per series: point estimates over all records after the cut, errors from n_bins
// equal bins over the first b * n_bins of them.
__global__ void __launch_bounds__(kAnaThreads) thermal_kernel(const double *series, int64_t len, int64_t cut,
                                                              int32_t n_bins, const double *T, const double *Nsites,
                                                              double *out) {
    __shared__ double sm[kAnaThreads / 32];
    __shared__ double s_bin[64][8];  // n_bins <= 64
    const int64_t sid = blockIdx.x;
    const double *h = series + sid * len * 4;
    const int64_t n = len - cut;
    const double Tt = T[sid], N = Nsites[sid];
    // reference shifts: the plain means of E and |M|
    double s0 = 0.0, s1 = 0.0;
    for (int64_t i = cut + threadIdx.x; i < len; i += blockDim.x) {
        const double *r = h + i * 4;
        s0 += r[0];
        s1 += sqrt(r[1] * r[1] + r[2] * r[2] + r[3] * r[3]);
    }
    const double Eref = block_sum(s0, sm) / (double)n;
    const double Aref = block_sum(s1, sm) / (double)n;
    double S[8];
    moment_sums(h, cut, len, Eref, Aref, sm, S);
    const int64_t b = n / n_bins;
    for (int k = 0; k < n_bins; ++k) {
        double Sk[8];
        moment_sums(h, cut + k * b, cut + (k + 1) * b, Eref, Aref, sm, Sk);
        if (threadIdx.x == 0)
            for (int q = 0; q < 8; ++q) s_bin[k][q] = Sk[q];
    }
    const double dn = (double)n;
    const double meanE = Eref + S[0] / dn, meanA = Aref + S[2] / dn, meanM2 = S[5] / dn;
    const double tau_e = tau_window(h, cut, n, 0, meanE, sm);
    const double tau_m = tau_window(h, cut, n, 1, meanA, sm);
    if (threadIdx.x != 0) return;
    double est[3];
    estimates(S, dn, N, Tt, est);
    const double covAE = S[4] / dn - (S[2] / dn) * (S[0] / dn);
    const double covM2E = S[7] / dn - meanM2 * (S[0] / dn);
    // the bin means' spread, and leave-one-bin-out (jackknife) estimates
    const double nb = (double)n_bins;
    double Tot[8] = {0.0, 0.0, 0.0, 0.0, 0.0, 0.0, 0.0, 0.0};
    double mbe = 0.0, mba = 0.0;
    for (int k = 0; k < n_bins; ++k) {
        for (int q = 0; q < 8; ++q) Tot[q] += s_bin[k][q];
        mbe += s_bin[k][0] / (double)b;
        mba += s_bin[k][2] / (double)b;
    }
    mbe /= nb;
    mba /= nb;
    double vbe = 0.0, vba = 0.0;
    for (int k = 0; k < n_bins; ++k) {
        const double de = s_bin[k][0] / (double)b - mbe, da = s_bin[k][2] / (double)b - mba;
        vbe += de * de;
        vba += da * da;
    }
    const double e_err = sqrt(vbe / (nb - 1.0)) / sqrt(nb) / N;
    const double m_err = sqrt(vba / (nb - 1.0)) / sqrt(nb) / N;
    double jm[3] = {0.0, 0.0, 0.0}, jv[3] = {0.0, 0.0, 0.0};
    const double nj = (double)((n_bins - 1) * b);
    for (int pass = 0; pass < 2; ++pass)  // mean of the jackknife estimates, then their spread
        for (int k = 0; k < n_bins; ++k) {
            double R[8], jk[3];
            for (int q = 0; q < 8; ++q) R[q] = Tot[q] - s_bin[k][q];
            estimates(R, nj, N, Tt, jk);  // shift-invariant forms: the sample's own means enter
            for (int q = 0; q < 3; ++q) {
                if (pass == 0)
                    jm[q] += jk[q] / nb;
                else
                    jv[q] += (jk[q] - jm[q]) * (jk[q] - jm[q]);
            }
        }
    double *o = out + sid * VEGAS_AVG_FIELDS;
    o[0] = meanE / N;
    o[1] = e_err;
    o[2] = meanA / N;
    o[3] = m_err;
    o[4] = est[0];
    o[5] = sqrt((nb - 1.0) / nb * jv[0]);
    o[6] = est[1];
    o[7] = sqrt((nb - 1.0) / nb * jv[1]);
    o[8] = est[2];
    o[9] = sqrt((nb - 1.0) / nb * jv[2]);
    o[10] = -covAE / meanA;
    o[11] = -covM2E / meanM2;
    o[12] = tau_e;
    o[13] = tau_m;
    o[14] = dn;
    o[15] = nb;
}

// ------------------------------------------------------------------ reweighting
// Bound by FP64 issue (two operations per SM and clock), which the exponentials filled: every exp
// is exp_int64 here, integer arithmetic only. tab: its table, copied into shared memory.
__device__ __forceinline__ void load_exp_table(unsigned long long *tab) {
    for (int k = threadIdx.x; k < 256; k += blockDim.x) tab[k] = kExp2Table[k];
    __syncthreads();
}

// D_i = ln sum_j n exp(-beta_j E_i - g_j) for every sample i.
__global__ void denom_kernel(const double *E, int64_t n_tot, const double *beta, const double *g, int32_t K,
                             double logn, double *D) {
    __shared__ unsigned long long tab[256];
    load_exp_table(tab);
    for (int64_t i = (int64_t)blockIdx.x * blockDim.x + threadIdx.x; i < n_tot; i += (int64_t)gridDim.x * blockDim.x) {
        const double e = E[i];
        double m = -INFINITY;
        for (int j = 0; j < K; ++j) m = fmax(m, -beta[j] * e - g[j]);
        double s = 0.0;
        for (int j = 0; j < K; ++j) s += exp_int64(-beta[j] * e - g[j] - m, tab);
        D[i] = logn + m + log(s);
    }
}

// Partial log-sum-exp of x_i = -beta E_i - D_i (and the x-weighted observables) per block:
// (max, sum of exp(x - max), sums of O exp(x - max)).
__global__ void __launch_bounds__(kAnaThreads) lse_kernel(const double *E, const double *D, const double *O,
                                                          int32_t n_obs, int64_t n_tot, const double *betas,
                                                          double *part) {
    __shared__ double sm[kAnaThreads / 32];
    __shared__ unsigned long long tab[256];
    load_exp_table(tab);
    const double beta = betas[blockIdx.y];
    const int64_t chunk = (n_tot + gridDim.x - 1) / gridDim.x;
    const int64_t i0 = (int64_t)blockIdx.x * chunk, i1 = min(n_tot, i0 + chunk);
    // the maximum by integer comparisons of the values' bits (mapped so that their order is the
    // values'): a comparison of doubles is an FP64 instruction
    auto ordered = [](long long v) { return v ^ ((v >> 63) & 0x7FFFFFFFFFFFFFFFLL); };
    long long mk = ordered(__double_as_longlong(-INFINITY));
    for (int64_t i = i0 + threadIdx.x; i < i1; i += blockDim.x) {
        const long long v = __double_as_longlong(-beta * E[i] - D[i]);
        if ((v & 0x7FFFFFFFFFFFFFFFLL) <= 0x7FF0000000000000LL) mk = max(mk, ordered(v));  // not NaN
    }
    double m = __longlong_as_double(ordered(mk));
    // block max (fixed order)
    for (int off = 16; off > 0; off >>= 1) m = fmax(m, __shfl_xor_sync(0xFFFFFFFFu, m, off));
    __shared__ double smax[kAnaThreads / 32];
    if ((threadIdx.x & 31) == 0) smax[threadIdx.x >> 5] = m;
    __syncthreads();
    double M = -INFINITY;
    for (int w = 0; w < kAnaThreads / 32; ++w) M = fmax(M, smax[w]);
    double s = 0.0, so[kMaxObs];
#pragma unroll
    for (int q = 0; q < kMaxObs; ++q) so[q] = 0.0;
    if (M > -INFINITY) {
        for (int64_t i = i0 + threadIdx.x; i < i1; i += blockDim.x) {
            const double w = exp_int64(-beta * E[i] - D[i] - M, tab);
            s += w;
#pragma unroll
            for (int q = 0; q < kMaxObs; ++q)
                if (q < n_obs) so[q] += w * O[i * n_obs + q];
        }
    }
    double *p = part + ((int64_t)blockIdx.y * gridDim.x + blockIdx.x) * (2 + kMaxObs);
    const double ts = block_sum(s, sm);
    double to[kMaxObs];
#pragma unroll
    for (int q = 0; q < kMaxObs; ++q)
        if (q < n_obs) to[q] = block_sum(so[q], sm);
    if (threadIdx.x == 0) {
        p[0] = M;
        p[1] = ts;
#pragma unroll
        for (int q = 0; q < kMaxObs; ++q)
            if (q < n_obs) p[2 + q] = to[q];
    }
}

// Combines the per-block partials of each row y, one warp per row (lanes over the blocks, then a
// butterfly): lse[y] = M + ln S and, when obs is not NULL, obs[y][q] = sum O exp(x) / sum exp(x).
__global__ void combine_kernel(const double *part, int32_t n_parts, int32_t n_rows, int32_t n_obs, double *lse,
                               double *obs) {
    const int y = (blockIdx.x * blockDim.x + threadIdx.x) >> 5, lane = threadIdx.x & 31;
    if (y >= n_rows) return;
    const double *p = part + (int64_t)y * n_parts * (2 + kMaxObs);
    double M = -INFINITY;
    for (int b = lane; b < n_parts; b += 32) M = fmax(M, p[b * (2 + kMaxObs)]);
    for (int off = 16; off > 0; off >>= 1) M = fmax(M, __shfl_xor_sync(0xFFFFFFFFu, M, off));
    double s = 0.0, so[kMaxObs];
#pragma unroll
    for (int q = 0; q < kMaxObs; ++q) so[q] = 0.0;
    for (int b = lane; b < n_parts; b += 32) {
        const double *pb = p + b * (2 + kMaxObs);
        if (pb[0] == -INFINITY) continue;
        const double f = exp(pb[0] - M);
        s += pb[1] * f;
#pragma unroll
        for (int q = 0; q < kMaxObs; ++q)
            if (q < n_obs) so[q] += pb[2 + q] * f;
    }
    for (int off = 16; off > 0; off >>= 1) {
        s += __shfl_xor_sync(0xFFFFFFFFu, s, off);
#pragma unroll
        for (int q = 0; q < kMaxObs; ++q)
            if (q < n_obs) so[q] += __shfl_xor_sync(0xFFFFFFFFu, so[q], off);
    }
    if (lane != 0) return;
    lse[y] = M + log(s);
    if (obs)
#pragma unroll
        for (int q = 0; q < kMaxObs; ++q)
            if (q < n_obs) obs[(int64_t)y * n_obs + q] = so[q] / s;
}

// State of the fixed-point iteration g_j <- ln sum_i exp(-beta_j E_i - D_i(g)), on the device.
struct MultiState {
    double diff;
    int32_t iters;    // iterations done
    uint32_t ticket;  // blocks done in the current one
    int32_t stop;     // 1: diff < tol, 2: a step the fused form cannot take (nothing was changed)
};

constexpr int kMultiRuns = 16;  // most runs of the fused form (a thread keeps two values per run)

// One iteration in one launch, for at most KM runs. With z_ij = -beta_j E_i - g_j the sample's
// denominator is n sum_j exp(z_ij), and the new g_j = g_j + ln sum_i a_ij / s_i - ln n with
// a_ij = exp(z_ij - z_ik), s_i = sum_j a_ij, k the sample's own run: the same K exponentials give
// the denominators and the sums, so none is taken twice and no logarithm per sample is left.
// A block takes a range of one run's samples (so z_ij - z_ik = db_j E_i + dg_j with its own few
// constants) and the last block combines the blocks' sums. Three FP64 operations per
// exponential and seven per sample remain. Values that leave the range of exp_int64, or a sum that
// underflows, stop the iteration unchanged (stop = 2) and the kernels above take that step.
// 8 runs x 20,011 samples: 364 us per iteration before (denom, lse and combine kernels with FP64
// exponentials, and a host synchronisation), 22.5 us now (half of it the FP64 pipe's share).
template <int KM>
__global__ void __launch_bounds__(kAnaThreads) multi_step_kernel(const double *E, int64_t n, int32_t K, const double *beta,
                                                                 double *g, double logn, double tol, double *part,
                                                                 MultiState *st) {
    __shared__ unsigned long long tab[256];
    __shared__ double s_db[KM], s_dg[KM];
    __shared__ double s_sum[KM][kAnaThreads + 8];
    __shared__ bool s_last;
    asm volatile("griddepcontrol.launch_dependents;" ::: "memory");
    const int k = blockIdx.y, tid = threadIdx.x;
    for (int q = tid; q < 256; q += kAnaThreads) tab[q] = kExp2Table[q];
    asm volatile("griddepcontrol.wait;" ::: "memory");
    if (__ldcg(&st->stop) != 0) return;
    if (tid < KM) {
        s_db[tid] = tid < K ? beta[k] - beta[tid] : 0.0;
        s_dg[tid] = tid < K ? __ldcg(g + k) - __ldcg(g + tid) : 0.0;
    }
    __syncthreads();
    double P[KM];
#pragma unroll
    for (int j = 0; j < KM; ++j) P[j] = 0.0;
    const int64_t chunk = (n + gridDim.x - 1) / gridDim.x, i0 = (int64_t)blockIdx.x * chunk, i1 = min(n, i0 + chunk);
    for (int64_t i = i0 + tid; i < i1; i += kAnaThreads) {
        const double e = E[(int64_t)k * n + i];
        double a[KM], s = 0.0;
#pragma unroll
        for (int j = 0; j < KM; ++j) {
            a[j] = 0.0;
            if (j < K) {
                a[j] = exp_int64(fma(s_db[j], e, s_dg[j]), tab);
                s += a[j];
            }
        }
        // 1 / s by Newton's iteration on the hardware's approximation (s >= 1; an infinite s leaves NaN)
        double r;
        asm("rcp.approx.ftz.f64 %0, %1;" : "=d"(r) : "d"(s));
        r = fma(r, fma(-s, r, 1.0), r);
        r = fma(r, fma(-s, r, 1.0), r);
#pragma unroll
        for (int j = 0; j < KM; ++j)
            if (j < K) P[j] = fma(a[j], r, P[j]);
    }
    // block sums with few FP64 instructions: threads' values through shared memory, kAnaThreads / KM
    // lanes per run adding KM each, then a butterfly over those lanes
    constexpr int L = kAnaThreads / KM;
#pragma unroll
    for (int j = 0; j < KM; ++j) s_sum[j][tid] = P[j];
    __syncthreads();
    {
        const int j = tid / L, l = tid % L;
        double v = 0.0;
        for (int q = l; q < kAnaThreads; q += L) v += s_sum[j][q];
        for (int off = (L < 32 ? L : 32) / 2; off > 0; off >>= 1) v += __shfl_xor_sync(0xFFFFFFFFu, v, off);
        __syncthreads();
        if (l % 32 == 0) s_sum[j][l / 32] = v;
        __syncthreads();
        if (tid < KM && tid < K) {
            double t = s_sum[tid][0];
            for (int q = 1; q < (L + 31) / 32; ++q) t += s_sum[tid][q];
            part[((int64_t)k * gridDim.x + blockIdx.x) * KM + tid] = t;
        }
    }
    __threadfence();
    __syncthreads();
    if (tid == 0) s_last = atomicAdd(&st->ticket, 1u) == gridDim.x * gridDim.y - 1u;
    __syncthreads();
    if (!s_last) return;
    __threadfence();
    // the last block: one warp per run adds the blocks' sums in order (lanes striding, a butterfly)
    const int n_part = gridDim.x * gridDim.y, lane = tid & 31;
    for (int j = tid >> 5; j < K; j += kAnaThreads / 32) {
        double v = 0.0;
        for (int b = lane; b < n_part; b += 32) v += __ldcg(part + (int64_t)b * KM + j);
        for (int off = 16; off > 0; off >>= 1) v += __shfl_xor_sync(0xFFFFFFFFu, v, off);
        if (lane == 0) s_sum[0][j] = v;
    }
    __syncthreads();
    if (tid < 32) {  // one lane per run (KM <= 16)
        const double sum = lane < K ? s_sum[0][lane] : 1.0, old = lane < K ? __ldcg(g + lane) : 0.0;
        const bool fine = sum > 1e-200 && sum < 1e200;
        double v = old + (log(sum) - logn);
        v -= __shfl_sync(0xFFFFFFFFu, v, 0);  // gauge: g_0 = 0
        double d = lane < K ? fabs(v - old) : 0.0;
        for (int off = 16; off > 0; off >>= 1) d = fmax(d, __shfl_xor_sync(0xFFFFFFFFu, d, off));
        const bool all = __all_sync(0xFFFFFFFFu, fine);
        if (all && lane < K) g[lane] = v;
        if (lane == 0) {
            st->ticket = 0;
            if (all) {
                st->diff = d;
                st->iters += 1;
            }
            st->stop = !all ? 2 : (d < tol ? 1 : 0);
        }
    }
}

// Device memory of one call: one allocation cut into 256-byte aligned pieces (an allocation and its
// release take about 20 us each). reserve() every piece, then allocate(), then take() them in order.
struct DevBuf {
    char *base = nullptr;
    size_t size = 0, used = 0;
    ~DevBuf() {
        if (base) cudaFree(base);
    }
    static size_t padded(size_t bytes) { return (bytes + 255) / 256 * 256; }
    void reserve(size_t bytes) { size += padded(bytes); }
    cudaError_t allocate() { return cudaMalloc((void **)&base, size > 0 ? size : 256); }
    template <typename T>
    T *take(size_t bytes) {
        T *p = (T *)(base + used);
        used += padded(bytes);
        return p;
    }
};

#define ACK(call)                                                                                        \
    do {                                                                                                 \
        cudaError_t e_ = (call);                                                                         \
        if (e_ != cudaSuccess)                                                                           \
            return ana_fail(e_ == cudaErrorMemoryAllocation ? VEGAS_ENOMEM : VEGAS_ECUDA,                \
                            std::string(#call) + ": " + cudaGetErrorString(e_));                         \
    } while (0)

vegas_status have_device() {
    int ndev = 0;
    cudaError_t e = cudaGetDeviceCount(&ndev);
    if (e != cudaSuccess || ndev == 0) return ana_fail(VEGAS_ECUDA, std::string("no CUDA device: ") + cudaGetErrorString(e));
    return VEGAS_OK;
}

}  // namespace

extern "C" const char *vegas_analysis_last_error(void) { return g_ana_err.c_str(); }

extern "C" vegas_status vegas_thermal_averages(const double *series, int64_t n_series, int64_t len, int64_t cut,
                                               int32_t n_bins, const double *T, const double *n_sites, double *out,
                                               void *cuda_stream) {
    try {
        if (!series || !T || !n_sites || !out) return ana_fail(VEGAS_EINVAL, "a required pointer is NULL");
        if (n_series < 1 || len < 1 || cut < 0 || cut >= len) return ana_fail(VEGAS_EINVAL, "need n_series >= 1 and 0 <= cut < len");
        if (n_bins < 2 || n_bins > 64) return ana_fail(VEGAS_EINVAL, "n_bins must be in [2, 64]");
        if ((len - cut) / n_bins < 1) return ana_fail(VEGAS_EINVAL, "fewer records after the cut than bins");
        if (n_series > INT32_MAX) return ana_fail(VEGAS_EINVAL, "too many series");
        for (int64_t s = 0; s < n_series; ++s)
            if (!(T[s] > 0.0) || !std::isfinite(T[s]) || !(n_sites[s] > 0.0))
                return ana_fail(VEGAS_EINVAL, "T and n_sites must be finite and > 0");
        vegas_status st = have_device();
        if (st != VEGAS_OK) return st;
        cudaStream_t stream = (cudaStream_t)cuda_stream;
        const size_t hb = sizeof(double) * 4 * (size_t)n_series * (size_t)len;
        const size_t sb = sizeof(double) * (size_t)n_series, ob = VEGAS_AVG_FIELDS * sb;
        DevBuf b;
        for (const size_t x : {hb, sb, sb, ob}) b.reserve(x);
        ACK(b.allocate());
        double *d_h = b.take<double>(hb), *d_T = b.take<double>(sb), *d_N = b.take<double>(sb), *d_out = b.take<double>(ob);
        ACK(cudaMemcpyAsync(d_h, series, hb, cudaMemcpyHostToDevice, stream));
        ACK(cudaMemcpyAsync(d_T, T, sizeof(double) * n_series, cudaMemcpyHostToDevice, stream));
        ACK(cudaMemcpyAsync(d_N, n_sites, sizeof(double) * n_series, cudaMemcpyHostToDevice, stream));
        thermal_kernel<<<(unsigned)n_series, kAnaThreads, 0, stream>>>(d_h, len, cut, n_bins, d_T, d_N, d_out);
        ACK(cudaGetLastError());
        ACK(cudaMemcpyAsync(out, d_out, sizeof(double) * VEGAS_AVG_FIELDS * n_series, cudaMemcpyDeviceToHost, stream));
        ACK(cudaStreamSynchronize(stream));
        return VEGAS_OK;
    } catch (...) {
        return analysis_host_exception();
    }
}

extern "C" vegas_status vegas_reweight(const double *E, const double *O, int32_t K, int64_t n, int32_t n_obs,
                                       const double *betas_k, const double *betas_out, int32_t n_out,
                                       int32_t max_iter, double tol, double *out, double *g_out, int32_t *iters_out,
                                       void *cuda_stream) {
    try {
        if (!E || !betas_k || (n_out > 0 && (!betas_out || !out)) || (n_obs > 0 && !O))
            return ana_fail(VEGAS_EINVAL, "a required pointer is NULL");
        if (K < 1 || n < 1 || n_obs < 0 || n_obs > kMaxObs || n_out < 0 || max_iter < 1 || !(tol > 0.0))
            return ana_fail(VEGAS_EINVAL, "need K >= 1, n >= 1, 0 <= n_obs <= 8, n_out >= 0, max_iter >= 1, tol > 0");
        const int64_t n_tot = (int64_t)K * n;
        for (int32_t k = 0; k < K; ++k)
            if (!std::isfinite(betas_k[k])) return ana_fail(VEGAS_EINVAL, "non-finite beta");
        int bad = 0;  // no early exit: the loop vectorises
        for (int64_t i = 0; i < n_tot; ++i) bad |= !(std::fabs(E[i]) <= 1.7976931348623157e308);
        if (bad) return ana_fail(VEGAS_EINVAL, "non-finite energy");
        vegas_status st = have_device();
        if (st != VEGAS_OK) return st;
        cudaStream_t stream = (cudaStream_t)cuda_stream;
        int dev = 0, sms = 1;
        ACK(cudaGetDevice(&dev));
        ACK(cudaDeviceGetAttribute(&sms, cudaDevAttrMultiProcessorCount, dev));
        const int parts = (int)std::min<int64_t>(256, (n_tot + kAnaThreads - 1) / kAnaThreads);
        // the averages' rows fill the GPU together: about eight blocks per SM over all of them, so that a
        // thread has many samples to a block sum (40 rows of 160,000: 540 us with 256 blocks per row)
        const int parts_out = std::max(1, std::min(parts, 8 * sms / std::max(n_out, 1)));
        const int rows = std::max<int32_t>(K, n_out);
        // fused iterations: two blocks per SM over all runs, at least kAnaThreads samples each
        const bool fused = K <= kMultiRuns;
        const int mx = (int)std::max<int64_t>(1, std::min<int64_t>(2 * sms / K, (n + kAnaThreads - 1) / kAnaThreads));
        const size_t D = sizeof(double), nb = D * (size_t)n_tot, kb = D * (size_t)K, tb = D * (size_t)std::max(n_out, 1);
        const size_t pb = D * std::max<size_t>((size_t)(2 + kMaxObs) * parts * rows, (size_t)mx * K * kMultiRuns);
        DevBuf b;
        for (const size_t x : {nb, nb * std::max(n_obs, 1), nb, kb, tb, kb, D * (size_t)rows, pb, tb * std::max(n_obs, 1),
                               sizeof(MultiState)})
            b.reserve(x);
        ACK(b.allocate());
        double *d_E = b.take<double>(nb), *d_O = b.take<double>(nb * std::max(n_obs, 1)), *d_D = b.take<double>(nb);
        double *d_bk = b.take<double>(kb), *d_bo = b.take<double>(tb), *d_g = b.take<double>(kb);
        double *d_lse = b.take<double>(D * (size_t)rows), *d_part = b.take<double>(pb);
        double *d_obs = b.take<double>(tb * std::max(n_obs, 1));
        MultiState *d_st = b.take<MultiState>(sizeof(MultiState));
        ACK(cudaMemcpyAsync(d_E, E, sizeof(double) * n_tot, cudaMemcpyHostToDevice, stream));
        if (n_obs > 0) ACK(cudaMemcpyAsync(d_O, O, sizeof(double) * n_tot * n_obs, cudaMemcpyHostToDevice, stream));
        ACK(cudaMemcpyAsync(d_bk, betas_k, sizeof(double) * K, cudaMemcpyHostToDevice, stream));
        if (n_out > 0) ACK(cudaMemcpyAsync(d_bo, betas_out, sizeof(double) * n_out, cudaMemcpyHostToDevice, stream));
        std::vector<double> g((size_t)K, 0.0), gn((size_t)K);
        ACK(cudaMemcpyAsync(d_g, g.data(), sizeof(double) * K, cudaMemcpyHostToDevice, stream));
        const double logn = std::log((double)n);
        const int dgrid = (int)std::min<int64_t>((n_tot + 255) / 256, 4096);
        auto combine = [&](int n_parts, int n_rows, int obs_, double *d_o) {
            combine_kernel<<<(n_rows + 3) / 4, 128, 0, stream>>>(d_part, n_parts, n_rows, obs_, d_lse, d_o);
        };
        MultiState ms{};
        ACK(cudaMemcpyAsync(d_st, &ms, sizeof ms, cudaMemcpyHostToDevice, stream));
        int32_t it = 0;  // iterations done
        bool done = false, general = !fused;
        while (!done && it < max_iter) {
            if (general) {  // one iteration by the separate kernels
                denom_kernel<<<dgrid, 256, 0, stream>>>(d_E, n_tot, d_bk, d_g, K, logn, d_D);
                lse_kernel<<<dim3(parts, K), kAnaThreads, 0, stream>>>(d_E, d_D, d_O, 0, n_tot, d_bk, d_part);
                combine(parts, K, 0, nullptr);
                ACK(cudaGetLastError());
                ACK(cudaMemcpyAsync(gn.data(), d_lse, sizeof(double) * K, cudaMemcpyDeviceToHost, stream));
                ACK(cudaStreamSynchronize(stream));
                double diff = 0.0;
                const double g0 = gn[0];
                for (int32_t k = 0; k < K; ++k) {
                    gn[(size_t)k] -= g0;  // gauge: g_0 = 0
                    diff = std::max(diff, std::fabs(gn[(size_t)k] - g[(size_t)k]));
                }
                if (!std::isfinite(diff))
                    return ana_fail(VEGAS_EDEVICE, "reweighting iteration produced a non-finite value");
                g = gn;
                ACK(cudaMemcpyAsync(d_g, g.data(), sizeof(double) * K, cudaMemcpyHostToDevice, stream));
                ++it;
                done = diff < tol;
                general = !fused;
                continue;
            }
            // a batch of fused iterations; those after the last one needed return at once
            ms = MultiState{0.0, it, 0u, 0};
            ACK(cudaMemcpyAsync(d_st, &ms, sizeof ms, cudaMemcpyHostToDevice, stream));
            cudaLaunchConfig_t cfg = {};
            cfg.gridDim = dim3((unsigned)mx, (unsigned)K);
            cfg.blockDim = dim3(kAnaThreads);
            cfg.stream = stream;
            cudaLaunchAttribute attr[1];
            attr[0].id = cudaLaunchAttributeProgrammaticStreamSerialization;
            attr[0].val.programmaticStreamSerializationAllowed = 1;
            cfg.attrs = attr;
            cfg.numAttrs = 1;
            const int batch = (int)std::min<int64_t>(kMultiBatch, max_iter - it);
            for (int q = 0; q < batch; ++q) {
                if (K <= 4)
                    ACK(cudaLaunchKernelEx(&cfg, multi_step_kernel<4>, (const double *)d_E, n, K, (const double *)d_bk, d_g,
                                           logn, tol, d_part, d_st));
                else if (K <= 8)
                    ACK(cudaLaunchKernelEx(&cfg, multi_step_kernel<8>, (const double *)d_E, n, K, (const double *)d_bk, d_g,
                                           logn, tol, d_part, d_st));
                else
                    ACK(cudaLaunchKernelEx(&cfg, multi_step_kernel<16>, (const double *)d_E, n, K, (const double *)d_bk, d_g,
                                           logn, tol, d_part, d_st));
            }
            ACK(cudaMemcpyAsync(&ms, d_st, sizeof ms, cudaMemcpyDeviceToHost, stream));
            ACK(cudaMemcpyAsync(g.data(), d_g, sizeof(double) * K, cudaMemcpyDeviceToHost, stream));
            ACK(cudaStreamSynchronize(stream));
            it = ms.iters;
            done = ms.stop == 1;
            general = ms.stop == 2;
            if (it > 0 && !general && !std::isfinite(ms.diff))
                return ana_fail(VEGAS_EDEVICE, "reweighting iteration produced a non-finite value");
        }
        if (g_out) std::memcpy(g_out, g.data(), sizeof(double) * K);
        if (iters_out) *iters_out = it;
        if (n_out > 0) {
            denom_kernel<<<dgrid, 256, 0, stream>>>(d_E, n_tot, d_bk, d_g, K, logn, d_D);
            lse_kernel<<<dim3(parts_out, n_out), kAnaThreads, 0, stream>>>(d_E, d_D, d_O, n_obs, n_tot, d_bo, d_part);
            combine(parts_out, n_out, n_obs, d_obs);
            ACK(cudaGetLastError());
            if (n_obs > 0)
                ACK(cudaMemcpyAsync(out, d_obs, sizeof(double) * n_out * n_obs, cudaMemcpyDeviceToHost, stream));
            ACK(cudaStreamSynchronize(stream));
        }
        return VEGAS_OK;
    } catch (...) {
        return analysis_host_exception();
    }
}
