// Analysis of a simulation history on the GPU: thermal averages with binned and jackknife
// errors, the Binder cumulant and the cumulants V1, V2, integrated autocorrelation times
// (Sec. II, Sec. IV.A-B), and single/multiple histogram reweighting (Sec. IV.E; Ferrenberg
// & Swendsen 1988, 1989). FP64 throughout; every sum is a fixed-order block reduction, so
// results do not change between runs.
#include <cooperative_groups.h>
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

// Sums over the block of the NQ values of every thread, in a fixed order, into out (shared memory),
// with few FP64 instructions (an FP64 instruction of a warp takes 64 cycles here, whatever its
// lanes do): warp w adds the threads' quantities w, w + 8, ... (a stride per lane, then a butterfly).
template <int NQ>
__device__ __forceinline__ void block_sums(const double (&v)[NQ], double (*sm)[kAnaThreads], double *out) {
    const int lane = threadIdx.x & 31;
#pragma unroll
    for (int q = 0; q < NQ; ++q) sm[q][threadIdx.x] = v[q];
    __syncthreads();
    for (int q = threadIdx.x >> 5; q < NQ; q += kAnaThreads / 32) {
        double s = 0.0;
#pragma unroll
        for (int k = 0; k < kAnaThreads / 32; ++k) s += sm[q][lane + 32 * k];
        for (int off = 16; off > 0; off >>= 1) s += __shfl_xor_sync(0xFFFFFFFFu, s, off);
        if (lane == 0) out[q] = s;
    }
    __syncthreads();
}

// Thermal averages run as four kernels over all series: |M| and the plain sums; centred values and
// moments per bin; estimates and errors; autocorrelation times. (One block per series with every
// step inside, |M| taken anew for every lag and the errors on one thread, took 4.4 ms for 64 series of
// 10,007 records, on 64 SMs and bound by their FP64 pipes; the whole call, with the 20 MB of records
// copied from the host, went from 5.1 to 0.59 ms.)
struct ThermalArgs {
    const double *series;  // [n_series][len][4]
    double *x;             // [2][n_series][stride]: E and |M| after the cut, then centred; zeros behind
    double *sums;          // [n_series][chunks][2]
    double *bins;          // [n_series][n_bins + 1][8], the last of the records behind the bins
    const double *T, *Nsites;
    double *out;           // [n_series][VEGAS_AVG_FIELDS]
    int64_t len, cut, n, stride, chunk;
    int32_t n_series, n_bins, chunks;
};

// |M| of every record after the cut, kept with E, and their sums over a chunk.
__global__ void __launch_bounds__(kAnaThreads) thermal_load_kernel(const ThermalArgs a) {
    __shared__ double sm[2][kAnaThreads], s_out[2];
    const int64_t sid = blockIdx.y;
    const double *h = a.series + (sid * a.len + a.cut) * 4;
    double *xe = a.x + sid * a.stride, *xa = a.x + (a.n_series + sid) * a.stride;
    const int64_t i0 = blockIdx.x * a.chunk, i1 = min(a.n, i0 + a.chunk);
    double v[2] = {0.0, 0.0};
    for (int64_t i = i0 + threadIdx.x; i < i1; i += kAnaThreads) {
        const double2 p = ((const double2 *)h)[2 * i], q = ((const double2 *)h)[2 * i + 1];
        const double m = sqrt(p.y * p.y + q.x * q.x + q.y * q.y);
        xe[i] = p.x;
        xa[i] = m;
        v[0] += p.x;
        v[1] += m;
    }
    block_sums<2>(v, sm, s_out);
    if (threadIdx.x < 2) a.sums[(sid * a.chunks + blockIdx.x) * 2 + threadIdx.x] = s_out[threadIdx.x];
}

// Mean of E and |M| over a series (the same in every block that asks).
__device__ __forceinline__ void series_means(const ThermalArgs &a, int64_t sid, double &Eref, double &Aref) {
    double v[2] = {0.0, 0.0};
    for (int k = threadIdx.x & 31; k < a.chunks; k += 32) {
        v[0] += a.sums[(sid * a.chunks + k) * 2];
        v[1] += a.sums[(sid * a.chunks + k) * 2 + 1];
    }
    for (int off = 16; off > 0; off >>= 1)
        for (int q = 0; q < 2; ++q) v[q] += __shfl_xor_sync(0xFFFFFFFFu, v[q], off);
    Eref = v[0] / (double)a.n;
    Aref = v[1] / (double)a.n;
}

// Centred values e' = E - Eref, a' = |M| - Aref of one bin (block n_bins: the records behind the
// bins), in place, and their moments: sums of e', e'^2, a', a'^2, a' e', M^2, M^4, M^2 e'. M^2 comes
// from the components, not from the rounded |M|.
__global__ void __launch_bounds__(kAnaThreads) thermal_bin_kernel(const ThermalArgs a) {
    __shared__ double sm[8][kAnaThreads], s_out[8], s_ref[2];
    const int64_t sid = blockIdx.y, b = a.n / a.n_bins;
    if (threadIdx.x < 32) {
        double e, m;
        series_means(a, sid, e, m);
        if (threadIdx.x == 0) {
            s_ref[0] = e;
            s_ref[1] = m;
        }
    }
    __syncthreads();
    const double Eref = s_ref[0], Aref = s_ref[1];
    double *xe = a.x + sid * a.stride, *xa = a.x + (a.n_series + sid) * a.stride;
    const double2 *h = (const double2 *)(a.series + (sid * a.len + a.cut) * 4);
    const bool rest = (int)blockIdx.x == a.n_bins;
    const int64_t i0 = blockIdx.x * b, i1 = rest ? a.n : i0 + b;
    double v[8] = {0.0, 0.0, 0.0, 0.0, 0.0, 0.0, 0.0, 0.0};
    for (int64_t i = i0 + threadIdx.x; i < i1; i += kAnaThreads) {
        const double2 p = h[2 * i], q = h[2 * i + 1];
        const double m2 = p.y * p.y + q.x * q.x + q.y * q.y, e = xe[i] - Eref, d = xa[i] - Aref;
        xe[i] = e;
        xa[i] = d;
        v[0] += e;
        v[1] += e * e;
        v[2] += d;
        v[3] += d * d;
        v[4] += d * e;
        v[5] += m2;
        v[6] += m2 * m2;
        v[7] += m2 * e;
    }
    if (rest)  // zeros behind the series: the lags read past its end
        for (int64_t i = a.n + threadIdx.x; i < a.stride; i += kAnaThreads) xe[i] = xa[i] = 0.0;
    block_sums<8>(v, sm, s_out);
    if (threadIdx.x < 8) a.bins[(sid * (a.n_bins + 1) + blockIdx.x) * 8 + threadIdx.x] = s_out[threadIdx.x];
}

// (c, chi, u4) from moment sums over n samples.
__device__ __forceinline__ void estimates(const double (&S)[8], double n, double N, double T, double (&out)[3]) {
    const double me = S[0] / n, ma = S[2] / n, m2 = S[5] / n;
    out[0] = (S[1] / n - me * me) / (N * T * T);
    out[1] = (S[3] / n - ma * ma) / (N * T);
    out[2] = 1.0 - (S[6] / n) / (3.0 * m2 * m2);
}

__device__ __forceinline__ double warp_sum(double v) {
    for (int off = 16; off > 0; off >>= 1) v += __shfl_xor_sync(0xFFFFFFFFu, v, off);
    return v;
}

// Point estimates over all records after the cut, errors from n_bins <= 64 equal bins (their spread
// and leave-one-bin-out jackknife estimates): one warp per series, a lane takes bins lane, lane + 32.
__global__ void thermal_estimate_kernel(const ThermalArgs a) {
    const int64_t sid = blockIdx.x;
    const int lane = threadIdx.x;
    const double *bins = a.bins + sid * (a.n_bins + 1) * 8;
    const double dn = (double)a.n, N = a.Nsites[sid], T = a.T[sid], nb = (double)a.n_bins;
    const double db = (double)(a.n / a.n_bins);
    double Eref, Aref;
    series_means(a, sid, Eref, Aref);
    double tot = 0.0;  // lane q < 8: quantity q over the bins
    if (lane < 8)
        for (int k = 0; k < a.n_bins; ++k) tot += bins[k * 8 + lane];
    const double all = lane < 8 ? tot + bins[a.n_bins * 8 + lane] : 0.0;
    double Tot[8], S[8];
#pragma unroll
    for (int q = 0; q < 8; ++q) {
        Tot[q] = __shfl_sync(0xFFFFFFFFu, tot, q);
        S[q] = __shfl_sync(0xFFFFFFFFu, all, q);
    }
    const double de = S[0] / dn, da = S[2] / dn, meanE = Eref + de, meanA = Aref + da, meanM2 = S[5] / dn;
    double est[3];
    estimates(S, dn, N, T, est);
    // bin means (their sums divided by the bins) and jackknife estimates of this lane's bins
    const double mbe = Tot[0] / db / nb, mba = Tot[2] / db / nb, nj = (double)((a.n_bins - 1) * (a.n / a.n_bins));
    double ve = 0.0, va = 0.0, jk[2][3], jm[3] = {0.0, 0.0, 0.0}, jv[3] = {0.0, 0.0, 0.0};
#pragma unroll
    for (int h = 0; h < 2; ++h) {
        const int k = lane + 32 * h;
        if (k >= a.n_bins) continue;
        const double xe = bins[k * 8] / db - mbe, xa = bins[k * 8 + 2] / db - mba;
        ve += xe * xe;
        va += xa * xa;
        double R[8];
#pragma unroll
        for (int q = 0; q < 8; ++q) R[q] = Tot[q] - bins[k * 8 + q];
        estimates(R, nj, N, T, jk[h]);  // shift-invariant forms: the sample's own means enter
#pragma unroll
        for (int q = 0; q < 3; ++q) jm[q] += jk[h][q];
    }
    ve = warp_sum(ve);
    va = warp_sum(va);
#pragma unroll
    for (int q = 0; q < 3; ++q) jm[q] = warp_sum(jm[q]) / nb;
#pragma unroll
    for (int h = 0; h < 2; ++h)
        if (lane + 32 * h < a.n_bins)
#pragma unroll
            for (int q = 0; q < 3; ++q) jv[q] += (jk[h][q] - jm[q]) * (jk[h][q] - jm[q]);
#pragma unroll
    for (int q = 0; q < 3; ++q) jv[q] = warp_sum(jv[q]);
    if (lane != 0) return;
    double *o = a.out + sid * VEGAS_AVG_FIELDS;
    const double jf = (nb - 1.0) / nb;
    o[0] = meanE / N;
    o[1] = sqrt(ve / (nb - 1.0)) / sqrt(nb) / N;
    o[2] = meanA / N;
    o[3] = sqrt(va / (nb - 1.0)) / sqrt(nb) / N;
    for (int q = 0; q < 3; ++q) {
        o[4 + 2 * q] = est[q];
        o[5 + 2 * q] = sqrt(jf * jv[q]);
    }
    o[10] = -(S[4] / dn - da * de) / meanA;
    o[11] = -(S[7] / dn - meanM2 * de) / meanM2;
    o[14] = dn;
    o[15] = nb;
}

constexpr int kLags = 16;  // lags per pass over the series

// Integrated autocorrelation time of E or |M|, Sokal's window (c = 6): a cluster of blocks per (series,
// quantity) takes kLags lags at a time (one multiply-add per record and lag, which bounds it; the
// centred series stays in L1), every block adds the cluster's sums in rank order, and all of them find
// the same window.
__global__ void __launch_bounds__(kAnaThreads) thermal_tau_kernel(const ThermalArgs a) {
    namespace cg = cooperative_groups;
    cg::cluster_group cl = cg::this_cluster();
    __shared__ double sm[kLags][kAnaThreads], s_blk[2][kLags];
    __shared__ double s_tau;
    __shared__ int s_done;
    const int CS = (int)cl.num_blocks(), rank = (int)cl.block_rank(), lane = threadIdx.x & 31;
    const int64_t idx = blockIdx.x / CS, which = idx & 1, sid = idx >> 1, n = a.n;
    double *x = a.x + (which * a.n_series + sid) * a.stride;
    const int64_t per = (n + CS - 1) / CS, i0 = rank * per, i1 = min(n, i0 + per);
    double v[kLags];
    auto total = [&](int buf) {  // lane q of a warp: the cluster's sum q, in rank order
        double t = 0.0;
        if (lane < kLags)
            for (int b = 0; b < CS; ++b) t += cl.map_shared_rank(&s_blk[buf][0], b)[lane];
        return t;
    };
    // The values were centred on the rounded plain mean: their own mean, added from the bins, goes too
    // (a constant series is 0 only then). Each block takes it off its own records; the barrier shows the
    // cluster's values to every block of it.
    double rest = 0.0;
    for (int b = lane; b <= a.n_bins; b += 32) rest += a.bins[(sid * (a.n_bins + 1) + b) * 8 + 2 * which];
    rest = warp_sum(rest) / (double)n;
#pragma unroll
    for (int q = 0; q < kLags; ++q) v[q] = 0.0;
    for (int64_t i = i0 + threadIdx.x; i < i1; i += kAnaThreads) {
        const double xi = x[i] - rest;
        x[i] = xi;
        v[0] += xi * xi;
    }
    block_sums<kLags>(v, sm, s_blk[0]);
    if (threadIdx.x == 0) {
        s_tau = 0.5;
        s_done = 0;
    }
    cl.sync();
    const double c0 = __shfl_sync(0xFFFFFFFFu, total(0), 0) / (double)n;
    int buf = 1;
    for (int64_t t0 = 1; t0 <= n / 2 && c0 != 0.0; t0 += kLags, buf ^= 1) {
#pragma unroll
        for (int q = 0; q < kLags; ++q) v[q] = 0.0;
        const int64_t e = min(i1, n - t0);
        for (int64_t i = i0 + threadIdx.x; i < e; i += kAnaThreads) {
            const double xi = x[i];
            const double *y = x + i + t0;  // zeros from n on
#pragma unroll
            for (int q = 0; q < kLags; ++q) v[q] = fma(xi, y[q], v[q]);
        }
        block_sums<kLags>(v, sm, s_blk[buf]);
        cl.sync();  // every block's sums are there (and nobody reads the other buffer any more)
        if (threadIdx.x < 32) {
            const int64_t t = t0 + lane;
            const bool in = lane < kLags && t <= n / 2;
            const double rho = in ? total(buf) / (double)(n - t) / c0 : 0.0;
            double run = s_tau, mine = run;  // partial sums in lag order
            for (int q = 0; q < kLags; ++q) {
                run += __shfl_sync(0xFFFFFFFFu, rho, q);
                if (lane == q) mine = run;
            }
            const uint32_t closed = __ballot_sync(0xFFFFFFFFu, in && (double)t >= 6.0 * mine);
            const double end = __shfl_sync(0xFFFFFFFFu, mine, closed ? __ffs(closed) - 1 : kLags - 1);
            if (lane == 0) {
                s_tau = end;
                s_done = closed != 0u;
            }
        }
        __syncthreads();
        if (s_done) break;
    }
    if (rank == 0 && threadIdx.x == 0) a.out[sid * VEGAS_AVG_FIELDS + 12 + which] = s_tau;
    cl.sync();  // no block leaves while another may read its sums
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
        int dev = 0, sms = 1;
        ACK(cudaGetDevice(&dev));
        ACK(cudaDeviceGetAttribute(&sms, cudaDevAttrMultiProcessorCount, dev));
        ThermalArgs a{};
        a.len = len;
        a.cut = cut;
        a.n = len - cut;
        a.n_series = (int32_t)n_series;
        a.n_bins = n_bins;
        a.stride = a.n + kLags;
        a.chunk = std::max<int64_t>(1024, (a.n + 63) / 64);
        a.chunks = (int32_t)((a.n + a.chunk - 1) / a.chunk);
        const size_t D = sizeof(double), ns = (size_t)n_series, hb = D * 4 * ns * (size_t)len, sb = D * ns;
        const size_t xb = D * 2 * ns * (size_t)a.stride, cb = D * 2 * ns * (size_t)a.chunks, bb = D * 8 * ns * (size_t)(n_bins + 1);
        const size_t ob = VEGAS_AVG_FIELDS * sb;
        DevBuf b;
        for (const size_t x : {hb, xb, cb, bb, sb, sb, ob}) b.reserve(x);
        ACK(b.allocate());
        double *d_h = b.take<double>(hb);
        a.series = d_h;
        a.x = b.take<double>(xb);
        a.sums = b.take<double>(cb);
        a.bins = b.take<double>(bb);
        double *d_T = b.take<double>(sb), *d_N = b.take<double>(sb), *d_out = b.take<double>(ob);
        a.T = d_T;
        a.Nsites = d_N;
        a.out = d_out;
        ACK(cudaMemcpyAsync(d_h, series, hb, cudaMemcpyHostToDevice, stream));
        ACK(cudaMemcpyAsync(d_T, T, sizeof(double) * n_series, cudaMemcpyHostToDevice, stream));
        ACK(cudaMemcpyAsync(d_N, n_sites, sizeof(double) * n_series, cudaMemcpyHostToDevice, stream));
        // series per launch: a grid's second dimension holds at most 65535
        for (int64_t s0 = 0; s0 < n_series; s0 += 65535) {
            ThermalArgs p = a;
            const unsigned m = (unsigned)std::min<int64_t>(65535, n_series - s0);
            p.n_series = (int32_t)n_series;  // rows of x between E and |M|
            p.series += s0 * len * 4;
            p.x += s0 * a.stride;
            p.sums += s0 * a.chunks * 2;
            p.bins += s0 * (n_bins + 1) * 8;
            p.T += s0;
            p.Nsites += s0;
            p.out += s0 * VEGAS_AVG_FIELDS;
            thermal_load_kernel<<<dim3((unsigned)a.chunks, m), kAnaThreads, 0, stream>>>(p);
            thermal_bin_kernel<<<dim3((unsigned)n_bins + 1u, m), kAnaThreads, 0, stream>>>(p);
            thermal_estimate_kernel<<<m, 32, 0, stream>>>(p);
            int cs = 1;  // blocks per cluster: as many as keep one block per SM, at most 8
            while (cs < 8 && (int64_t)m * 2 * (cs * 2) <= sms) cs *= 2;
            cudaLaunchConfig_t cfg = {};
            cfg.gridDim = dim3(m * 2u * (unsigned)cs);
            cfg.blockDim = dim3(kAnaThreads);
            cfg.stream = stream;
            cudaLaunchAttribute attr[1];
            attr[0].id = cudaLaunchAttributeClusterDimension;
            attr[0].val.clusterDim.x = (unsigned)cs;
            attr[0].val.clusterDim.y = 1;
            attr[0].val.clusterDim.z = 1;
            cfg.attrs = attr;
            cfg.numAttrs = 1;
            ACK(cudaLaunchKernelEx(&cfg, thermal_tau_kernel, p));
        }
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
