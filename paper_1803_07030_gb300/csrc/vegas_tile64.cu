// The tiled cooperative sweep in FP64 (uniform trials): parts, mailbox words and records as in
// vegas_tile.cu, every step of an attempt as pass64_kernel's, so the oracle's spins bit for bit.
//
// What bounds a small FP64 sample: an FP64 instruction of a warp takes 64 cycles on GB300 (19 per
// warp instruction over an SM with four warps), however few of its lanes are active, and an attempt
// on one lane is a chain of about 190 of them (12 us per colour class). So the chain is cut to
// what has to follow the neighbours' spins, and laid across lanes:
//  - six lanes per site (x, y, z of the field and of its part over lower colours), five sites per
//    warp: 16 FP64 instructions per class for rows of six links. The field still adds its links one
//    by one in row order;
//  - trials and acceptance uniforms depend on no spin: warps of their own draw them up to four
//    classes ahead (one site per lane; the uniforms' conversions are exact in integers);
//  - the decision u < exp(-beta dE) is taken in FP32 when the two sides differ by more than FP32's
//    error bound, in FP64 as before otherwise (about one attempt in a million);
//  - energy shares and sums run after the spin is on its way.
// 8^3 ferromagnet: 24.2 us per MCS with grid barriers and one lane per site, 4.4 now.
#include <cuda_runtime.h>

#include <algorithm>
#include <cstdint>
#include <vector>

#include "vegas_fp64.cuh"
#include "vegas_internal.h"
#include "vegas_tile.cuh"
#include "vegas_tile.h"

namespace vegas {
namespace {

constexpr int kBarSweep = 1, kBarFull = 2, kBarEmpty = 4;  // as in vegas_tile.cu
constexpr unsigned kAll = 0xFFFFFFFFu;

__device__ __forceinline__ float as_f(uint32_t x) { return __uint_as_float(x); }

// Whether a wait of one part of the block for another has run out at its n-th poll: that part may
// itself wait timeout_ns for a remote word, so after twice that and a second.
__device__ __forceinline__ bool inner_wait_over(uint32_t n, uint64_t &since, int64_t timeout_ns) {
    if ((n & 1023u) != 0) return false;
    const uint64_t now = tile_ns();
    if (since == 0) since = now;
    return (now - since) / 2 > (uint64_t)timeout_ns + 500000000u;
}

// W: links per fixed row (6 or kEllRow; padded with links of J = 0 to the site itself). PM: 0 no
// anisotropy and uniform parameters, else 2.
template <int W, int PM>
__global__ void __launch_bounds__(kTile64Threads + kTile64Trial + 32) tile64_kernel(const Tile64Args ta) {
    extern __shared__ __align__(16) unsigned char smem[];
    const TileArgs &tt = ta.t;
    const PassArgs &a = tt.pass;
    const int NT = (int)blockDim.x - kTile64Trial - 32, tid = (int)threadIdx.x, lane = tid & 31;
    const int r = (int)blockIdx.x / tt.P, part = (int)blockIdx.x - r * tt.P, R = 1 << a.log2R;
    if ((int)blockIdx.x == tt.skip_block) return;  // fault injection: this block never stores a word
    const TilePart pt = tt.parts[part];
    const int nc = tt.n_colours, cap = tt.cap;
    double *sp = (double *)smem;                               // [3][cap]
    double *s_J = (double *)(smem + ta.J_off);                 // [own][W]
    Tile64Trial *s_trial = (Tile64Trial *)(smem + ta.trial_off);  // [kTile64Ahead][widest]
    double *s_part = (double *)(smem + tt.part_off);           // [2][E, M][NT]
    uint32_t *s_cnt = (uint32_t *)(s_part + 4 * NT);           // [2][NT]
    uint32_t *s_idx = (uint32_t *)(smem + tt.rows_off);        // [own][W]
    uint32_t *s_orig = (uint32_t *)(smem + tt.orig_off);
    int32_t *s_pub = (int32_t *)(smem + tt.pub_off), *s_slot = (int32_t *)(smem + tt.slot_off);
    TileClass *s_cls = (TileClass *)(smem + tt.cls_off);
    __shared__ volatile int s_ok;                       // 0: every warp leaves
    __shared__ volatile int s_ready[kTile64Ahead];      // classes drawn into a trial slot: sequence + 1
    __shared__ volatile int s_used;                     // classes whose trials are no longer needed
    RunState *rs = a.run;
    const uint32_t t0 = rs->t, rec0 = rs->rec;
    if (tid == 0) {
        s_ok = *(volatile uint32_t *)tt.abort == 0u ? 1 : 0;
        s_used = 0;
    }
    if (tid < kTile64Ahead) s_ready[tid] = 0;
    for (int c = tid; c < nc; c += blockDim.x) s_cls[c] = tt.classes[part * nc + c];
    const double4_32a *S = (const double4_32a *)a.spins;
    for (int k = tid; k < pt.n_own + pt.n_halo; k += blockDim.x) {
        const int g = __ldg(tt.site + pt.site_begin + k);
        const double4_32a v = S[(int64_t)g * R + r];
        sp[k] = v.x;
        sp[cap + k] = v.y;
        sp[2 * cap + k] = v.z;
        if (k < pt.n_own) {
            s_orig[k] = (uint32_t)__ldg(tt.orig + pt.own_begin + k);
            s_pub[k] = __ldg(tt.pub + pt.own_begin + k);
        } else {
            s_slot[k - pt.n_own] = __ldg(tt.halo_slot + pt.halo_begin + k - pt.n_own);
        }
    }
    for (int k = tid; k < pt.n_own * W; k += blockDim.x) {
        s_idx[k] = __ldg((const uint32_t *)tt.rows + (int64_t)pt.own_begin * W + k);
        s_J[k] = __ldg(ta.J + (int64_t)pt.own_begin * W + k);
    }
    __syncthreads();
    if (s_ok == 0) return;  // a wait of an earlier launch of the run ran out
    const uint32_t inst = (uint32_t)(a.inst0 + r);
    const uint32_t k0 = (uint32_t)a.seed, k1 = (uint32_t)(a.seed >> 32);
    if (tid >= NT + kTile64Trial) {
        // the record warp: totals of every MCS over the sweeping threads, in a fixed order. Lane roles
        // as in the sweep: lanes 6 s + 2 c hold component c of the magnetization.
        const int role = lane < 30 && (lane % 6) % 2 == 0 ? (lane % 6) / 2 : -1;
        for (int m = 0; m < tt.mcs; ++m) {
            const int b = m & 1;
            bar_sync(kBarFull + b, NT + 32);
            if (s_ok == 0) return;
            double e = 0.0, v = 0.0;
            uint32_t n = 0;
            for (int k = lane; k < NT; k += 32) {
                e += s_part[(b * 2) * NT + k];
                v += s_part[(b * 2 + 1) * NT + k];
                n += s_cnt[b * NT + k];
            }
            bar_arrive(kBarEmpty + b, NT + 32);
            // one butterfly for E over all lanes; the magnetization's lanes of one component are 6 apart
            for (int off = 16; off > 0; off >>= 1) e += __shfl_xor_sync(kAll, e, off);
            double mq = v;
            for (int s = 1; s < 5; ++s) mq += __shfl_sync(kAll, v, lane % 6 + 6 * s);
            n = __reduce_add_sync(kAll, n);
            const int64_t at = ((int64_t)m << a.log2R) + r;
            if (lane == 0) {
                tt.partial[(at * 4) * tt.P + part] = e;  // [mcs][R][4][P]
                tt.count[at * tt.P + part] = n;
            }
            if (lane < 6 && role >= 0) tt.partial[(at * 4 + 1 + role) * tt.P + part] = mq;
        }
        return;
    }
    if (tid >= NT) {
        // trial warps: class after class, kTile64Trial / 32 warps in turn, at most kTile64Ahead classes
        // ahead of the sweep
        const int w = (tid - NT) >> 5;
        const int64_t total = (int64_t)tt.mcs * nc;
        for (int64_t seq = w; seq < total; seq += kTile64Trial / 32) {
            int go = 1;
            uint64_t since = 0;
            if (lane == 0)  // one lane waits for all: they leave together
                for (uint32_t n = 1; go && (int)seq - s_used >= kTile64Ahead; ++n) {
                    if (s_ok == 0) {
                        go = 0;
                    } else if (inner_wait_over(n, since, tt.timeout_ns)) {  // the sweeping warps give up in turn
                        atomicOr(a.err, kErrTimeout);
                        go = 0;
                    } else {
                        __nanosleep(40);
                    }
                }
            __syncwarp();
            if (!__shfl_sync(kAll, go, 0)) return;
            const int c = (int)(seq % nc), slot = (int)(seq % kTile64Ahead);
            const uint32_t t = t0 + (uint32_t)(seq / nc);
            const TileClass cl = s_cls[c];
            for (int k = cl.begin + lane; k < cl.end; k += 32) {
                const uint32_t orig = s_orig[k];
                double sn = a.u64.s;
                if (PM == 2 && a.params_mode == 2)
                    sn = ((const double4_32a *)a.p0)[__ldg(tt.site + pt.site_begin + k)].w;
                const double3 u = sphere64(orig, t, inst, kPurposeTrial64, k0, k1, a.err);
                const uint4 wa = philox10(make_uint4(orig, t, inst, kPurposeAccept64), k0, k1);
                Tile64Trial &o = s_trial[slot * ta.widest + k - cl.begin];
                const bool one = __double_as_longlong(sn) == 0x3FF0000000000000LL;  // 1 x = x exactly
                o.x = one ? u.x : dm(sn, u.x);
                o.y = one ? u.y : dm(sn, u.y);
                o.z = one ? u.z : dm(sn, u.z);
                o.u = ((unsigned long long)wa.x << 21) | (unsigned long long)(wa.y >> 11);
            }
            __threadfence_block();
            __syncwarp();
            if (lane == 0) s_ready[slot] = (int)seq + 1;
        }
        return;
    }
    // ---- sweeping warps: lane 6 s + 2 c + h of a warp holds, for its site s, component c of the field
    // (h = 0) or of its part over lower colours (h = 1)
    const uint32_t step = rec0 / rs->mcs;
    const double *sc = rs->sched + ((int64_t)step * a.n_inst + a.inst_local0 + r) * 2;
    const double beta = sc[0], B = sc[1];
    const float betaf = (float)beta;
    const bool act = lane < 30;
    const int s5 = act ? lane / 6 : 4, base = 6 * s5, comp = act ? (lane - base) >> 1 : 2, h = lane & 1;
    const int per_round = (NT >> 5) * 5, my = (tid >> 5) * 5 + s5;
    float4 *mail = tt.mail + (int64_t)r * tt.n_mail * 2;
    const double un = comp == 0 ? a.u64.nx : comp == 1 ? a.u64.ny : a.u64.nz;
    const double Bn_uniform = dm(B, un);
    double accE = 0.0, accM = 0.0;
    uint32_t nacc = 0;
    bool nan_seen = false;
    // everything of an attempt that no other site's sweep changes
    struct Prep {
        uint32_t idx[W / 2];
        double J[W / 2], S, P, d, Bn, dan, dcub, kk, an_new, an_old, cub_new, cub_old;
        uint32_t lower, orig;
        int32_t pub;
        unsigned long long u;
    } q{};
    auto prep = [&](int k, const TileClass &cl, int slot) {
        q.orig = s_orig[k];
        q.pub = s_pub[k];
        q.lower = 0u;
#pragma unroll
        for (int j = 0; j < W; ++j) q.lower |= (s_idx[k * W + j] >> 16) << j;
#pragma unroll
        for (int j = 0; j < W / 2; ++j) {
            q.idx[j] = s_idx[k * W + 2 * j + h] & 0xFFFFu;
            q.J[j] = s_J[k * W + 2 * j + h];
        }
        const Tile64Trial &tr = s_trial[slot * ta.widest + k - cl.begin];
        q.P = comp == 0 ? tr.x : comp == 1 ? tr.y : tr.z;
        q.u = tr.u;
        q.S = sp[comp * cap + k];
        q.d = ds(q.P, q.S);
        q.Bn = Bn_uniform;
    };
    // the anisotropy terms of the prepared sites (all lanes of a warp take part)
    auto prep_aniso = [&](int k, bool has) {
        double e = comp == 0 ? a.u64.ex : comp == 1 ? a.u64.ey : a.u64.ez, kc = a.u64.kc;
        q.kk = a.u64.k;
        if (a.params_mode == 2 && has) {
            const int g = __ldg(tt.site + pt.site_begin + k);
            const double4_32a p0 = ((const double4_32a *)a.p0)[g], p1 = ((const double4_32a *)a.p1)[g];
            q.Bn = dm(B, comp == 0 ? p0.x : comp == 1 ? p0.y : p0.z);
            e = comp == 0 ? p1.x : comp == 1 ? p1.y : p1.z;
            q.kk = p1.w;
            kc = ((const double *)a.pk)[g];
        }
        // lanes h = 0: of the trial, h = 1: of the present spin
        const double v = h == 0 ? q.P : q.S, ve = dm(v, e);
        const double p = da(da(__shfl_sync(kAll, ve, base + h), __shfl_sync(kAll, ve, base + 2 + h)),
                            __shfl_sync(kAll, ve, base + 4 + h));
        const double pp = dm(p, p), vv = dm(v, v);
        const double xx = __shfl_sync(kAll, vv, base + h), yy = __shfl_sync(kAll, vv, base + 2 + h),
                     zz = __shfl_sync(kAll, vv, base + 4 + h);
        const double cub = da(da(dm(xx, yy), dm(yy, zz)), dm(xx, zz));
        q.an_new = __shfl_sync(kAll, pp, base);
        q.an_old = __shfl_sync(kAll, pp, base + 1);
        q.cub_new = dm(kc, __shfl_sync(kAll, cub, base));
        q.cub_old = dm(kc, __shfl_sync(kAll, cub, base + 1));
        q.dan = -dm(q.kk, ds(q.an_new, q.an_old));
        q.dcub = -dm(kc, ds(__shfl_sync(kAll, cub, base), __shfl_sync(kAll, cub, base + 1)));
    };
    // all lanes of a warp take part
    auto finish = [&](int k, bool has, uint32_t t) {
        double prod[W / 2];
#pragma unroll
        for (int j = 0; j < W / 2; ++j) prod[j] = has ? dm(q.J[j], sp[comp * cap + (int)q.idx[j]]) : 0.0;
        double f = 0.0;  // links in row order
#pragma unroll
        for (int j = 0; j < W; ++j) {
            const double v = __shfl_sync(kAll, prod[j / 2], base + 2 * comp + (j & 1));
            if (h == 0 || ((q.lower >> j) & 1u)) f = da(f, v);
        }
        const double dh = dm(q.d, da(f, q.Bn));  // lanes h = 0
        const double dEex = -da(da(__shfl_sync(kAll, dh, base), __shfl_sync(kAll, dh, base + 2)), __shfl_sync(kAll, dh, base + 4));
        const double dE = PM == 0 ? dEex : da(da(dEex, q.dan), q.dcub);
        const long long bits = __double_as_longlong(dE);
        const bool nan = (bits & 0x7FFFFFFFFFFFFFFFLL) > 0x7FF0000000000000LL;
        const bool ok = accept64(bits, dE, beta, betaf, q.u) && !nan;
        // the spin goes out first, in two words: (x, y low, tag) and (y high, z, tag)
        const double n = ok ? q.P : q.S;
        const uint32_t lo = (uint32_t)__double2loint(n), hi = (uint32_t)__double2hiint(n);
        const uint32_t ylo = __shfl_sync(kAll, lo, base + 2), yhi = __shfl_sync(kAll, hi, base + 2);
        if (!has) return;
        if (h == 0) {
            if (q.pub >= 0 && comp == 0) mail_store(mail + 2 * (int64_t)q.pub, as_f(lo), as_f(hi), as_f(ylo), t + 1u);
            if (q.pub >= 0 && comp == 2) mail_store(mail + 2 * (int64_t)q.pub + 1, as_f(yhi), as_f(lo), as_f(hi), t + 1u);
            sp[comp * cap + k] = n;
            accM += n;
        }
        accE = fma(-n, h == 0 ? q.Bn : f, accE);  // -S.(B n) and -S.(lower field), one term per lane
        if (lane == base) {
            if (PM != 0) accE -= q.kk * (ok ? q.an_new : q.an_old) + (ok ? q.cub_new : q.cub_old);
            nan_seen |= nan;
            nacc += ok ? 1u : 0u;
            if (a.alog && t < a.alog_mcs)
                a.alog[(int64_t)t * a.alog_stride + a.alog_base + (int64_t)r * a.n_sample_sites + q.orig] = ok ? 1 : 0;
        }
    };
    // the remote spins [h0, h1) of one class after the MCS with this tag, into shared memory (false: the
    // wait ran out, here or in another block)
    auto collect = [&](int h0, int h1, uint32_t tag) -> bool {
        for (int i = h0 + tid; i < h1; i += NT) {
            const float4 *p = mail + 2 * (int64_t)s_slot[i];
            float4 v0 = mail_load(p), v1 = mail_load(p + 1);
            uint64_t since = 0;
            for (uint32_t n = 1; __float_as_uint(v0.w) != tag || __float_as_uint(v1.w) != tag; ++n) {
                if ((n & 255u) == 0) {
                    const uint64_t now = tile_ns();
                    if (since == 0) since = now;
                    if (*(volatile uint32_t *)tt.abort) return false;
                    if ((int64_t)(now - since) > tt.timeout_ns) {
                        atomicOr(a.err, kErrTimeout);
                        atomicExch(tt.abort, 1u);
                        return false;
                    }
                }
                if (__float_as_uint(v0.w) != tag) v0 = mail_load(p);
                if (__float_as_uint(v1.w) != tag) v1 = mail_load(p + 1);
            }
            const int k = pt.n_own + i;
            sp[k] = __hiloint2double((int)__float_as_uint(v0.y), (int)__float_as_uint(v0.x));
            sp[cap + k] = __hiloint2double((int)__float_as_uint(v1.x), (int)__float_as_uint(v0.z));
            sp[2 * cap + k] = __hiloint2double((int)__float_as_uint(v1.z), (int)__float_as_uint(v1.y));
        }
        return true;
    };
    int pend = -1, seq = 0;
    for (int m = 0; m < tt.mcs; ++m) {
        const uint32_t t = t0 + (uint32_t)m;
        for (int c = 0; c < nc; ++c, ++seq) {
            const TileClass cl = s_cls[c];
            const int slot = seq % kTile64Ahead;
            bool drawn = true;  // the trial warps run classes ahead
            if (s_ready[slot] != seq + 1) {
                uint64_t since = 0;
                for (uint32_t n = 1; drawn && s_ready[slot] != seq + 1; ++n) drawn = !inner_wait_over(n, since, tt.timeout_ns);
                if (!drawn) atomicOr(a.err, kErrTimeout);
            }
            __threadfence_block();
            const int n_cls = cl.end - cl.begin;
            int j = my;
            bool has = act && j < n_cls;
            if (has) prep(cl.begin + j, cl, slot);
            if (PM != 0) prep_aniso(cl.begin + j, has);
            {
                const bool ok = drawn && (pend < 0 || collect(s_cls[pend].halo_begin, s_cls[pend].halo_end, pend < c ? t + 1u : t));
                // the class before is final in this block, with its remote spins
                if (!bar_and(kBarSweep, NT, ok)) {  // every thread leaves, and the other warps with them
                    s_ok = 0;
                    bar_arrive(kBarFull + (m & 1), NT + 32);
                    return;
                }
                if (tid == 0) s_used = seq;  // every warp is done with the class before
            }
            for (int j0 = 0; j0 < n_cls; j0 += per_round) {
                finish(cl.begin + j, has, t);
                j += per_round;
                has = act && j < n_cls;
                if (j0 + per_round < n_cls) {
                    if (has) prep(cl.begin + j, cl, slot);
                    if (PM != 0) prep_aniso(cl.begin + j, has);
                }
            }
            pend = c;
        }
        const int b = m & 1;
        if (m >= 2) bar_sync(kBarEmpty + b, NT + 32);
        s_part[(b * 2) * NT + tid] = act ? accE : 0.0;
        s_part[(b * 2 + 1) * NT + tid] = act && h == 0 ? accM : 0.0;
        s_cnt[b * NT + tid] = nacc;
        bar_arrive(kBarFull + b, NT + 32);
        accE = accM = 0.0;
        nacc = 0;
    }
    bar_sync(kBarSweep, NT);
    for (int k = tid; k < pt.n_own; k += NT)
        ((double4_32a *)a.spins)[(int64_t)__ldg(tt.site + pt.site_begin + k) * R + r] =
            make_double4_32a(sp[k], sp[cap + k], sp[2 * cap + k], 0.0);
    if (nan_seen) atomicOr(a.err, kErrNaN);
}

using Tile64Fn = void (*)(Tile64Args);

Tile64Fn select_tile64(const Tile64Args &a) {
    const bool plain = a.t.pass.params_mode == 0;
    if (a.t.width == 6) return plain ? tile64_kernel<6, 0> : tile64_kernel<6, 2>;
    return plain ? tile64_kernel<kEllRow, 0> : tile64_kernel<kEllRow, 2>;
}

}  // namespace

int tile64_shape(Tile64Args &ta, const TileShape &s, TilePlan &p, std::vector<double> &J, size_t *smem) {
    TileArgs &a = ta.t;
    int dev = 0, most = 0;
    if (cudaGetDevice(&dev) != cudaSuccess ||
        cudaDeviceGetAttribute(&most, cudaDevAttrMaxSharedMemoryPerBlockOptin, dev) != cudaSuccess)
        return 0;
    int own = 1;
    for (const TileClass &cl : p.classes) own = std::max(own, cl.end - cl.begin);
    if (own > kTile64Sites) return 0;  // larger shares fill the lanes of the other sweeps
    // one round of five sites per warp, as far as the block's warps go
    const int warps = std::min(kTile64Threads / 32, (own + 4) / 5), nt = 32 * warps;
    ta.widest = own;
    auto align = [](size_t x) { return (x + 15) / 16 * 16; };
    const int W = a.width;
    a.cap = p.max_loc;
    size_t at = align((size_t)a.cap * 24);
    ta.J_off = (int32_t)at;
    at = align(at + (size_t)p.max_own * W * 8);
    ta.trial_off = (int32_t)at;
    at = align(at + (size_t)kTile64Ahead * own * sizeof(Tile64Trial));
    a.part_off = (int32_t)at;
    at = align(at + (size_t)nt * (4 * 8 + 2 * 4));
    a.rows_off = (int32_t)at;
    at = align(at + (size_t)p.max_own * W * 4);
    a.orig_off = (int32_t)at;
    at = align(at + (size_t)p.max_own * 4);
    a.pub_off = (int32_t)at;
    at = align(at + (size_t)p.max_own * 4);
    a.slot_off = (int32_t)at;
    at = align(at + (size_t)p.max_halo * 4);
    a.cls_off = (int32_t)at;
    *smem = align(at + (size_t)a.n_colours * sizeof(TileClass));
    const Tile64Fn f = select_tile64(ta);
    cudaFuncAttributes fa;
    int nb = 0;
    // the limit belongs to the kernel, which other contexts launch too: raised to the device's
    if (cudaFuncGetAttributes(&fa, f) != cudaSuccess || *smem + fa.sharedSizeBytes > (size_t)most ||
        cudaFuncSetAttribute(f, cudaFuncAttributeMaxDynamicSharedMemorySize, most - (int)fa.sharedSizeBytes) != cudaSuccess ||
        cudaOccupancyMaxActiveBlocksPerMultiprocessor(&nb, f, nt + kTile64Trial + 32, *smem) != cudaSuccess || nb < 1)
        return 0;
    // words of (local site | lower flag << 16), and J beside them
    a.n_codes = 0;
    tile_tables(a, s, p);
    const int2 *pairs = (const int2 *)p.rows.get();  // the FP32 J of a pair is not used
    J.assign((size_t)s.n * W, 0.0);
    std::vector<uint32_t> idx((size_t)s.n * W);
    for (int32_t q = 0; q < s.parts; ++q)
        for (int32_t k = 0; k < p.parts[(size_t)q].n_own; ++k) {
            const size_t row = (size_t)(p.parts[(size_t)q].own_begin + k);
            const int32_t g = p.own[(size_t)q][(size_t)k];
            for (int w = 0; w < W; ++w) idx[row * W + w] = (uint32_t)pairs[row * W + w].x;
            for (int64_t e = s.row_ptr[g]; e < s.row_ptr[g + 1]; ++e) J[row * W + (size_t)(e - s.row_ptr[g])] = s.J[e];
        }
    p.row_bytes = idx.size() * 4;
    std::copy(idx.begin(), idx.end(), (uint32_t *)p.rows.get());
    return nt;
}

int launch_tile64(const Tile64Args &a, int threads, size_t smem, void *stream) {
    cudaStream_t st = (cudaStream_t)stream;
    const TileArgs &t = a.t;
    // no word may carry a tag of this launch before it is stored (the MCS counter can be set back)
    cudaError_t e = cudaMemsetAsync(t.mail, 0, ((size_t)t.n_mail << t.pass.log2R) * 2 * sizeof(float4), st);
    if (e != cudaSuccess) return (int)e;
    cudaLaunchConfig_t cfg = {};
    cfg.gridDim = dim3((unsigned)(t.P << t.pass.log2R));
    cfg.blockDim = dim3((unsigned)(threads + kTile64Trial + 32));
    cfg.dynamicSmemBytes = smem;
    cfg.stream = st;
    cudaLaunchAttribute attr[1];
    attr[0].id = cudaLaunchAttributeCooperative;
    attr[0].val.cooperative = 1;
    cfg.attrs = attr;
    cfg.numAttrs = 1;
    if ((e = cudaLaunchKernelEx(&cfg, select_tile64(a), a)) != cudaSuccess) return (int)e;
    return launch_tile_record(t, stream);
}

}  // namespace vegas
