// Tiled cooperative sweep of one FP32 sample: the sample is cut into parts of compact regions,
// and one block per (part, replica) keeps its part's spins (and, as they fit, links and site
// ids) in shared memory for every MCS of the launch. Blocks exchange only the spins of boundary
// sites, each through a 16-byte mailbox word that carries the MCS it belongs to.
//
// What bounds a small sample's sweep is the chain through the colour classes of an MCS: with
// one grid barrier per class and neighbour spins in L2, a class cost two to three L2 round trips
// and an atomic per block on one counter. Here a class costs one L2 trip: a boundary spin is
// stored as one 128-bit word (x, y, z, tag) right after its attempt, and the blocks that read it
// poll that very word, so no flag, fence or barrier stands between the data and its reader;
// sites without a remote reader are swept while the words travel, and the next attempt's random
// numbers, trial and links are prepared before the wait. The MCS's FP64 totals are formed by four
// warps of their own, from two shared-memory buffers in turn: an FP64 instruction of a warp takes
// 64 cycles here however few lanes are active (19 per warp instruction over an SM), so a shuffle
// tree in every sweeping warp took 2 us per MCS and one record warp for all four sums still 0.3 us
// per 32 threads. Large parts are bound by instruction issue (112 cycles per 32 attempts).
//
// us per MCS, before (grid barriers, neighbours in L2) and now: 64^3 with uniaxial anisotropy
// 17.5 and 4.9, the 29k-site core/shell particle 23.0 and 4.8, a 13k-site fcc sphere x 8 replicas
// 23.5 and 5.3, 128^3 54.6 and 25.8.
//
// Why one mailbox word per site is enough: tag t + 1 marks the value after MCS t. Site i of part
// N (class c) is read by part b because some site j of b (class c') links to i; then N reads j.
// N overwrites i's word in MCS t + 1 only after it has read j's word of class c' for that
// sweep, and b stored that word after it had read i's word of MCS t (b reads every remote word
// of class c before it attempts any site of the next class). So no word is overwritten unread.
//
// All blocks are co-resident (cooperative launch) and every wait is bounded by timeout_ns.
#include <cuda_runtime.h>

#include <algorithm>
#include <atomic>
#include <cmath>
#include <cstdint>
#include <cstdlib>
#include <cstring>
#include <exception>
#include <memory>
#include <mutex>
#include <new>
#include <thread>
#include <vector>

#include "vegas_device.cuh"
#include "vegas_internal.h"
#include "vegas_tile.cuh"
#include "vegas_tile.h"

namespace vegas {
namespace {

// Named barriers: the sweeping threads among themselves; the two partial-sum buffers between
// them and the record warp (full: the sums are written, empty: the record warp has read them).
constexpr int kBarSweep = 1, kBarFull = 2, kBarEmpty = 4;

// Everything of an attempt that no other site's sweep changes.
template <int W, int FMT>
struct TilePrep {
    uint32_t orig, wacc;
    int32_t pub;  // mailbox word, or -1
    Site32 p;
    float4 Si;
    float3 P;
    TileRow<W, FMT> row;
};

// W: links per fixed row (6 or kEllRow; shorter rows are padded with links of J = 0 to the site
// itself, which add signed zeros). PM: 0 uniform parameters without anisotropy, 3 no cubic
// anisotropy, 2 any. MEM: what a block
// keeps in shared memory beside the spins: 2 rows, site ids and remote words' indices, 1 the ids
// and indices, 0 nothing (the rest is read through L1 from tables in the block's own order). FMT 1
// halves the rows (samples of at most kTileCodes exchange values): for parts whose rows do not fit
// otherwise, or are read from L2 (128^3, 100 MB of pairs: 46.8 us per MCS, 29.1 with words; 27.5 once
// the warps added their sums, which left room for 512 threads in place of 384; 25.8 without compensated
// sums. There it is bound by the latency of an attempt with 16 sweeping warps per SM (issue 45%): kTileThreads
// and their registers are the limit, a warp takes 36 bytes of shared memory beside 12 per spin. Slower, against
// 27.5 to 28.8: rows fetched a round ahead 30.9, two sites in flight per thread 30.5; rows by link pair the same).
template <int W, int POL, int PM, int MEM, int FMT>
__global__ void __launch_bounds__(kTileThreads + kTileRecord) tile32_kernel(const TileArgs ta) {
    extern __shared__ __align__(16) unsigned char smem[];
    const PassArgs &a = ta.pass;
    const int NT = (int)blockDim.x - kTileRecord, tid = (int)threadIdx.x;
    const int r = (int)blockIdx.x / ta.P, part = (int)blockIdx.x - r * ta.P, R = 1 << a.log2R;
    if ((int)blockIdx.x == ta.skip_block) return;  // fault injection: this block never stores a word
    const TilePart pt = ta.parts[part];
    const int nc = ta.n_colours, cap = ta.cap;
    // shared memory: spins, rows, site ids, remote words' indices, class bounds, partial sums
    float *sp = (float *)smem;
    TileRow<W, FMT> *s_rows = (TileRow<W, FMT> *)(smem + ta.rows_off);
    float *s_J = (float *)(smem + ta.code_off);
    uint32_t *s_orig = (uint32_t *)(smem + ta.orig_off);
    int32_t *s_pub = (int32_t *)(smem + ta.pub_off);
    int32_t *s_slot = (int32_t *)(smem + ta.slot_off);
    TileClass *s_cls = (TileClass *)(smem + ta.cls_off);
    // one or two buffers of [E, Mx, My, Mz][NT], and of [NT] counts
    float *s_part = (float *)(smem + ta.part_off);
    uint32_t *s_cnt = (uint32_t *)(s_part + (1 + ta.two_buffers) * 4 * NT);
    // MEM 0: the warps' sums, [4][NT / 32] in FP64 and [NT / 32] counts
    double *s_sum = (double *)(smem + ta.part_off);
    uint32_t *s_num = (uint32_t *)(s_sum + 4 * (NT >> 5));
    __shared__ int s_ok;  // 0: the record warp leaves
    RunState *rs = a.run;
    const uint32_t t0 = rs->t, rec0 = rs->rec;
    if (tid == 0) s_ok = *(volatile uint32_t *)ta.abort == 0u ? 1 : 0;
    for (int c = tid; c < nc; c += blockDim.x) s_cls[c] = ta.classes[part * nc + c];
    const float4 *S = (const float4 *)a.spins;
    for (int k = tid; k < pt.n_own + pt.n_halo; k += blockDim.x) {
        const int g = __ldg(ta.site + pt.site_begin + k);
        const float4 v = S[(int64_t)g * R + r];
        loc_set(sp, cap, k, v.x, v.y, v.z);
        if (MEM >= 1 && k < pt.n_own) {
            s_orig[k] = (uint32_t)__ldg(ta.orig + pt.own_begin + k);
            s_pub[k] = __ldg(ta.pub + pt.own_begin + k);
        }
        if (MEM >= 1 && k >= pt.n_own) s_slot[k - pt.n_own] = __ldg(ta.halo_slot + pt.halo_begin + k - pt.n_own);
    }
    const TileRow<W, FMT> *g_rows = (const TileRow<W, FMT> *)ta.rows + pt.own_begin;
    if (MEM == 2)
        for (int k = tid; k < pt.n_own * (W / 2); k += blockDim.x)
            s_rows[k / (W / 2)].q[k % (W / 2)] = __ldg(&g_rows[0].q[0] + k);
    if (FMT == 1)
        for (int k = tid; k < ta.n_codes; k += blockDim.x) s_J[k] = ta.codes[k];
    __syncthreads();
    if (s_ok == 0) return;  // a wait of an earlier launch of the run ran out
    if (tid >= NT) {
        // record warp q: the total of quantity q over the sweeping threads after every MCS, in a
        // fixed order in FP64 (and, in warp 0, the accepted attempts)
        const int lane = tid & 31, q = (tid - NT) >> 5;
        for (int m = 0; m < ta.mcs; ++m) {
            const int b = m & ta.two_buffers;
            bar_sync(kBarFull + b, NT + kTileRecord);
            if (s_ok == 0) return;
            double v = 0.0;
            uint32_t n = 0;
            if (MEM == 0) {
                if (lane < (NT >> 5)) {
                    v = s_sum[q * (NT >> 5) + lane];
                    if (q == 0) n = s_num[lane];
                }
            } else {
                const float *x = s_part + (b * 4 + q) * NT;
                for (int k = lane; k < NT; k += 32) v += (double)x[k];
                if (q == 0)
                    for (int k = lane; k < NT; k += 32) n += s_cnt[b * NT + k];
            }
            bar_arrive(kBarEmpty + b, NT + kTileRecord);
            for (int off = 16; off > 0; off >>= 1) v += __shfl_xor_sync(0xFFFFFFFFu, v, off);
            const int64_t at = ((int64_t)m << a.log2R) + r;
            if (lane == 0) ta.partial[(at * 4 + q) * ta.P + part] = v;  // [mcs][R][4][P]
            if (q == 0) {
                n = __reduce_add_sync(0xFFFFFFFFu, n);
                if (lane == 0) ta.count[at * ta.P + part] = n;
            }
        }
        return;
    }
    const uint32_t step = rec0 / rs->mcs;
    const double *sc = rs->sched + ((int64_t)step * a.n_inst + a.inst_local0 + r) * 2;
    const float beta = (float)sc[0], B = (float)sc[1];
    const uint32_t inst = (uint32_t)(a.inst0 + r);
    float4 *mail = ta.mail + (int64_t)r * ta.n_mail;
    bool nan_seen = false;
    auto prep = [&](int k, uint32_t t, TilePrep<W, FMT> &q) {
        q.orig = MEM >= 1 ? s_orig[k] : (uint32_t)__ldg(ta.orig + pt.own_begin + k);
        q.pub = MEM >= 1 ? s_pub[k] : __ldg(ta.pub + pt.own_begin + k);
        q.Si = loc_spin(sp, cap, k);
#pragma unroll
        for (int j = 0; j < W / 2; ++j) q.row.q[j] = MEM == 2 ? s_rows[k].q[j] : __ldg(&g_rows[k].q[j]);
        int g = 0;
        if (PM != 0 || POL) g = __ldg(ta.site + pt.site_begin + k);
        q.p = Site32{a.u32.nx, a.u32.ny, a.u32.nz, a.u32.s, a.u32.ex, a.u32.ey, a.u32.ez, a.u32.k, a.u32.kc};
        if (PM != 0 && a.params_mode == 2) q.p = site_params32(a, 2, g);
        uint4 rw = make_uint4(q.orig, t, inst, kPurposeTrial32);
#pragma unroll
        for (int j = 0; j < 10; ++j) {  // Philox with the round keys as kernel arguments
            const uint32_t lo0 = 0xD2511F53u * rw.x, hi0 = __umulhi(0xD2511F53u, rw.x);
            const uint32_t lo1 = 0xCD9E8D57u * rw.z, hi1 = __umulhi(0xCD9E8D57u, rw.z);
            rw = make_uint4(hi1 ^ rw.y ^ ta.rk0[j], lo1, hi0 ^ rw.w ^ ta.rk1[j], lo0);
        }
        q.P = POL ? policy_trial32(a.pol32[g], 0.f, q.Si, q.p.sn, rw) : trial_random32(rw, q.p.sn);
        q.wacc = rw.z;
    };
    // the thread's sums of E and Mz, Mx and My over the MCS
    float2 fem = make_float2(0.f, 0.f), fxy = fem;
    uint32_t nacc = 0;
    auto finish = [&](int k, uint32_t t, const TilePrep<W, FMT> &q, const TileClass &cl) {
        // the field in row order (l: its part over lower colours)
        float2 hxy = make_float2(0.f, 0.f), lxy = make_float2(0.f, 0.f);
        float hz = 0.f, lz = 0.f;
        if (cl.lower_mode == 2) {
#pragma unroll
            for (int j = 0; j < W; ++j)
                link32(loc_spin(sp, cap, q.row.site(j)), q.row.J(j, s_J), q.row.lower(j), hxy, hz, lxy, lz);
        } else {
#pragma unroll
            for (int j = 0; j < W; ++j)
                link32(loc_spin(sp, cap, q.row.site(j)), q.row.J(j, s_J), false, hxy, hz, lxy, lz);
            if (cl.lower_mode == 1) {  // every link goes to a lower colour
                lxy = hxy;
                lz = hz;
            }
        }
        float4 Sn;
        bool ok, bad;
        float e;
        attempt32<PM, 2>(q.Si, hxy, hz, lxy, lz, q.p, beta, B, q.P, q.wacc, Sn, ok, e, bad);
        if (q.pub >= 0) mail_store(mail + q.pub, Sn.x, Sn.y, Sn.z, t + 1u);
        if (ok) loc_set(sp, cap, k, Sn.x, Sn.y, Sn.z);
        nan_seen |= bad;
        nacc += ok ? 1u : 0u;
        fem = __fadd2_rn(fem, make_float2(e, Sn.z));
        fxy = __fadd2_rn(fxy, make_float2(Sn.x, Sn.y));
        if (a.alog && t < a.alog_mcs)
            a.alog[(int64_t)t * a.alog_stride + a.alog_base + (int64_t)r * a.n_sample_sites + q.orig] = ok ? 1 : 0;
    };
    // the remote words [h0, h1) of one class after the MCS with this tag, into shared memory
    // (false: the wait ran out, here or in another block)
    auto collect = [&](int h0, int h1, uint32_t tag) -> bool {
        for (int h = h0 + tid; h < h1; h += 2 * NT) {  // two words in flight per thread
            const bool two = h + NT < h1;
            const int32_t *slot = MEM >= 1 ? s_slot : ta.halo_slot + pt.halo_begin;
            const float4 *p0 = mail + slot[h], *p1 = mail + slot[two ? h + NT : h];
            float4 v0 = mail_load(p0), v1 = mail_load(p1);
            uint64_t since = 0;
            for (uint32_t n = 1; __float_as_uint(v0.w) != tag || __float_as_uint(v1.w) != tag; ++n) {
                if ((n & 255u) == 0) {
                    const uint64_t now = tile_ns();
                    if (since == 0) since = now;
                    if (*(volatile uint32_t *)ta.abort) return false;
                    if ((int64_t)(now - since) > ta.timeout_ns) {
                        atomicOr(a.err, kErrTimeout);
                        atomicExch(ta.abort, 1u);
                        return false;
                    }
                }
                if (__float_as_uint(v0.w) != tag) v0 = mail_load(p0);
                if (__float_as_uint(v1.w) != tag) v1 = mail_load(p1);
            }
            loc_set(sp, cap, pt.n_own + h, v0.x, v0.y, v0.z);
            if (two) loc_set(sp, cap, pt.n_own + h + NT, v1.x, v1.y, v1.z);
        }
        return true;
    };
    int pend = -1;  // the class whose remote words have not been read yet
    for (int m = 0; m < ta.mcs; ++m) {
        const uint32_t t = t0 + (uint32_t)m;
        for (int c = 0; c < nc; ++c) {
            const TileClass cl = s_cls[c];
            int k = cl.begin + tid;
            TilePrep<W, FMT> q;
            if (k < cl.end) prep(k, t, q);
            if (pend >= 0) {
                const bool ok = collect(s_cls[pend].halo_begin, s_cls[pend].halo_end, pend < c ? t + 1u : t);
                // the class before is final in this block, with its remote spins
                if (!bar_and(kBarSweep, NT, ok)) {  // every thread leaves, and the record warp with them
                    s_ok = 0;
                    bar_arrive(kBarFull + (m & ta.two_buffers), NT + kTileRecord);
                    return;
                }
            }
            while (k < cl.end) {
                finish(k, t, q, cl);
                k += NT;
                if (k < cl.end) prep(k, t, q);
            }
            pend = c;
        }
        // this MCS's sums of every thread (at most 64 attempts each) to the record warp
        const int b = m & ta.two_buffers;
        if (MEM == 0) {
            // long parts: shared memory goes to spins, so each warp adds its threads' sums, in FP64; the
            // first two steps halve the quantities per lane (six additions for the four)
            const int lane = tid & 31;
            const double v[4] = {(double)fem.x, (double)fxy.x, (double)fxy.y, (double)fem.y};
            const bool hi = lane & 16, odd = lane & 8;
            double x = (hi ? v[2] : v[0]) + __shfl_xor_sync(0xFFFFFFFFu, hi ? v[0] : v[2], 16);
            double y = (hi ? v[3] : v[1]) + __shfl_xor_sync(0xFFFFFFFFu, hi ? v[1] : v[3], 16);
            x = (odd ? y : x) + __shfl_xor_sync(0xFFFFFFFFu, odd ? x : y, 8);
            for (int off = 4; off > 0; off >>= 1) x += __shfl_xor_sync(0xFFFFFFFFu, x, off);
            const uint32_t n = __reduce_add_sync(0xFFFFFFFFu, nacc);
            if (m > 0) bar_sync(kBarEmpty, NT + kTileRecord);
            if ((lane & 7) == 0) s_sum[(lane >> 3) * (NT >> 5) + (tid >> 5)] = x;
            if (lane == 0) s_num[tid >> 5] = n;
            bar_arrive(kBarFull, NT + kTileRecord);
            fem = fxy = make_float2(0.f, 0.f);
            nacc = 0;
            continue;
        }
        if (m > ta.two_buffers) bar_sync(kBarEmpty + b, NT + kTileRecord);
        float *o = s_part + b * 4 * NT + tid;
        o[0] = fem.x;
        o[NT] = fxy.x;
        o[2 * NT] = fxy.y;
        o[3 * NT] = fem.y;
        s_cnt[b * NT + tid] = nacc;
        bar_arrive(kBarFull + b, NT + kTileRecord);
        fem = fxy = make_float2(0.f, 0.f);
        nacc = 0;
    }
    bar_sync(kBarSweep, NT);
    for (int k = tid; k < pt.n_own; k += NT) {
        const float4 v = loc_spin(sp, cap, k);
        ((float4 *)a.spins)[(int64_t)__ldg(ta.site + pt.site_begin + k) * R + r] = v;
    }
    if (nan_seen) atomicOr(a.err, kErrNaN);
}

// The records of a launch's MCS: one warp per (MCS, replica) adds the parts' totals in a fixed
// order (lanes striding over the parts, a butterfly).
__global__ void tile_record_kernel(const TileArgs ta) {
    const PassArgs &a = ta.pass;
    const RunState *rs = a.run;
    const int64_t w = ((int64_t)blockIdx.x * blockDim.x + threadIdx.x) >> 5;
    const int lane = threadIdx.x & 31, r = (int)(w & ((1 << a.log2R) - 1));
    const int64_t m = w >> a.log2R;
    if (m >= ta.mcs) return;
    double v[4];
#pragma unroll
    for (int q = 0; q < 4; ++q) {
        v[q] = 0.0;
        for (int b = lane; b < ta.P; b += 32) v[q] += ta.partial[(w * 4 + q) * ta.P + b];
    }
    uint32_t n = 0;
    for (int b = lane; b < ta.P; b += 32) n += ta.count[w * ta.P + b];
    for (int off = 16; off > 0; off >>= 1) {
#pragma unroll
        for (int q = 0; q < 4; ++q) v[q] += __shfl_xor_sync(0xFFFFFFFFu, v[q], off);
    }
    n = __reduce_add_sync(0xFFFFFFFFu, n);
    if (lane == 0) {
        const int64_t at = ((int64_t)rs->rec + m) * a.n_inst + a.inst_local0 + r;
#pragma unroll
        for (int q = 0; q < 4; ++q) rs->hist[at * 4 + q] = v[q];
        if (rs->acc_hist) rs->acc_hist[at] = n;
    }
}

using TileFn = void (*)(TileArgs);

template <int W, int MEM>
TileFn select_w(const TileArgs &a) {
    if (a.pass.pol32) return tile32_kernel<W, 1, 2, MEM, 0>;
    if (a.cubic) return tile32_kernel<W, 0, 2, MEM, 0>;
    if (a.pass.params_mode == 0) return a.n_codes ? tile32_kernel<W, 0, 0, MEM, 1> : tile32_kernel<W, 0, 0, MEM, 0>;
    return a.n_codes ? tile32_kernel<W, 0, 3, MEM, 1> : tile32_kernel<W, 0, 3, MEM, 0>;
}

template <int W>
TileFn select_mem(const TileArgs &a) {
    return a.mem == 2 ? select_w<W, 2>(a) : a.mem == 1 ? select_w<W, 1>(a) : select_w<W, 0>(a);
}

TileFn select_tile(const TileArgs &a) { return a.width == 6 ? select_mem<6>(a) : select_mem<kEllRow>(a); }

}  // namespace

namespace {

// f(part, scratch) for every part, on several host threads; scratch: n words of the thread, 0 at
// first. An exception in a thread is passed on.
template <typename F>
void for_parts(int32_t parts, int32_t n, F &&f) {
    const int nt = (int)std::min<int64_t>({(int64_t)parts, (int64_t)std::max(1u, std::thread::hardware_concurrency()), 16,
                                           (int64_t)n / 4096 + 1});
    std::atomic<int32_t> next(0);
    std::exception_ptr err;
    std::mutex mu;
    auto work = [&] {
        try {
            // calloc: a thread's parts touch few pages of it
            std::unique_ptr<uint32_t, void (*)(void *)> scratch((uint32_t *)std::calloc((size_t)n, sizeof(uint32_t)), std::free);
            if (!scratch) throw std::bad_alloc();
            for (int32_t p; (p = next.fetch_add(1)) < parts;) f(p, scratch.get());
        } catch (...) {
            std::lock_guard<std::mutex> lk(mu);
            err = std::current_exception();
        }
    };
    std::vector<std::thread> th;
    try {
        for (int k = 1; k < nt; ++k) th.emplace_back(work);
    } catch (...) {  // fewer threads do
    }
    work();
    for (std::thread &t : th) t.join();
    if (err) std::rethrow_exception(err);
}

// First site of part p in class c. With `columns` a part takes the same range of places in every
// class; otherwise each class's equal share.
int32_t share(const TileShape &s, const TilePlan &out, int32_t c, int64_t p) {
    const int64_t nc = s.cstart[c + 1] - s.cstart[c], w = out.columns ? out.widest : nc;
    return s.cstart[c] + (int32_t)std::min(nc, (p * w + s.parts - 1) / s.parts);
}

}  // namespace

// Parts of compact regions: ranges of each class in memory order (a Morton curve when the sample
// gives positions). When a part's share of a class is one round of threads, a part takes the
// same places in every class and thread k of a block the k-th: it then adds the FP32 shares of
// site w of every class, in class order, as a thread of every sweep with a thread per site of the class
// does, and the histories agree with that sweep's to the FP64 sums' rounding.
bool tile_plan(const TileShape &s, TilePlan &out) {
    const int32_t n = s.n, nc = s.n_colours, P = s.parts;
    if (P < 1 || nc < 1) return false;
    out = TilePlan();
    for (int32_t c = 0; c < nc; ++c) out.widest = std::max(out.widest, s.cstart[c + 1] - s.cstart[c]);
    // one round per class: the order of a class's sites within it does not matter for speed
    const bool one_round = ((int64_t)out.widest + P - 1) / P + 1 <= kTileThreads;
    out.columns = one_round;
    out.part.resize((size_t)n);
    out.local.resize((size_t)n);
    out.word.resize((size_t)n);
    for (int32_t p = 0; p < P; ++p)
        for (int32_t c = 0; c < nc; ++c)
            std::fill(out.part.begin() + share(s, out, c, p), out.part.begin() + share(s, out, c, p + 1), p);
    out.classes.resize((size_t)P * nc);
    out.parts.resize((size_t)P);
    out.own.resize((size_t)P);
    out.halo.resize((size_t)P);
    for (int32_t p = 0, at = 0; p < P; ++p) {
        out.parts[(size_t)p].own_begin = at;
        for (int32_t c = 0; c < nc; ++c) {
            TileClass &cl = out.classes[(size_t)p * nc + c];
            cl.begin = at - out.parts[(size_t)p].own_begin;
            at += share(s, out, c, p + 1) - share(s, out, c, p);
            cl.end = at - out.parts[(size_t)p].own_begin;
            cl.lower_mode = s.lower_mode[c];
        }
        out.parts[(size_t)p].n_own = at - out.parts[(size_t)p].own_begin;
        out.max_own = std::max(out.max_own, out.parts[(size_t)p].n_own);
    }
    // own sites in order (several rounds: those with a remote reader first, to store their words
    // early) and the remote sites each part reads, class by class
    for_parts(P, n, [&](int32_t p, uint32_t *mark) {
        std::vector<int32_t> &o = out.own[(size_t)p], late;
        std::vector<std::vector<int32_t>> h((size_t)nc);
        o.reserve((size_t)out.parts[(size_t)p].n_own);
        int32_t words = 0;
        for (int32_t c = 0; c < nc; ++c) {
            late.clear();
            const int32_t g1 = share(s, out, c, p + 1);
            for (int32_t g = share(s, out, c, p); g < g1; ++g) {
                bool pub = false;
                for (int64_t e = s.row_ptr[g]; e < s.row_ptr[g + 1]; ++e) {
                    const int32_t j = s.col[e];
                    if (out.part[(size_t)j] == p) continue;
                    pub = true;
                    if (mark[j] == (uint32_t)p + 1u) continue;
                    mark[j] = (uint32_t)p + 1u;
                    h[(size_t)(std::upper_bound(s.cstart, s.cstart + nc + 1, j) - s.cstart) - 1].push_back(j);
                }
                out.word[(size_t)g] = pub ? words++ : -1;  // counted from the part's first
                if (pub || one_round) {
                    out.local[(size_t)g] = (int32_t)o.size();
                    o.push_back(g);
                } else {
                    late.push_back(g);
                }
            }
            for (int32_t g : late) {
                out.local[(size_t)g] = (int32_t)o.size();
                o.push_back(g);
            }
        }
        out.parts[(size_t)p].n_words = words;
        std::vector<int32_t> &halo = out.halo[(size_t)p];
        for (int32_t c = 0; c < nc; ++c) {
            TileClass &cl = out.classes[(size_t)p * nc + c];
            cl.halo_begin = (int32_t)halo.size();
            halo.insert(halo.end(), h[(size_t)c].begin(), h[(size_t)c].end());
            cl.halo_end = (int32_t)halo.size();
        }
    });
    int32_t halos = 0;
    for (int32_t p = 0; p < P; ++p) {
        TilePart &pt = out.parts[(size_t)p];
        pt.n_halo = (int32_t)out.halo[(size_t)p].size();
        pt.halo_begin = halos;
        halos += pt.n_halo;
        pt.site_begin = pt.own_begin + pt.halo_begin;
        pt.word_begin = out.n_mail;
        out.n_mail += pt.n_words;
        out.max_halo = std::max(out.max_halo, pt.n_halo);
        out.max_loc = std::max(out.max_loc, pt.n_own + pt.n_halo);
    }
    return out.max_loc <= 65535;
}

void host_ranges(int64_t n, int32_t chunks, const std::function<void(int64_t, int64_t)> &f) {
    if (n < 1) return;
    if (chunks <= 1) return f(0, n);
    for_parts(chunks, chunks * 4096, [&](int32_t q, uint32_t *) { f(n * q / chunks, n * (q + 1) / chunks); });
}

void exchange_values(const double *J, int64_t n_links, std::vector<float> &values) {
    auto add = [](std::vector<float> &to, float v) {
        if (to.size() <= (size_t)kTileCodes && std::find(to.begin(), to.end(), v) == to.end()) to.push_back(v);
    };
    auto scan = [&](std::vector<float> &to, int64_t e0, int64_t e1) {
        double a = NAN, b = NAN;  // two values seen: a glass has two, in random order
        for (int64_t e = e0; e < e1; ++e)
            if ((J[e] != a) & (J[e] != b)) {
                add(to, (float)J[e]);
                b = a;
                a = J[e];
            }
    };
    const int32_t chunks = (int32_t)std::min<int64_t>(16, n_links / (1 << 19) + 1);  // a thread costs 0.05 ms
    std::vector<std::vector<float>> got((size_t)chunks);
    host_ranges(chunks, chunks, [&](int64_t q, int64_t) { scan(got[(size_t)q], n_links * q / chunks, n_links * (q + 1) / chunks); });
    for (const auto &x : got)
        for (float v : x) add(values, v);
    add(values, 0.0f);
}

namespace {

// The block's tables: sites, ids, words, and the rows in local site numbers, as pairs or
// (a.n_codes) words.
void write_tables(const TileArgs &a, const TileShape &s, TilePlan &p) {
    const int W = a.width;
    p.row_bytes = (size_t)s.n * W * (a.n_codes ? 4 : 8);
    p.rows.reset(new unsigned char[p.row_bytes + 16]);
    const TilePart &last = p.parts[(size_t)s.parts - 1];
    p.halo_slot.resize((size_t)(last.halo_begin + last.n_halo));
    p.site.resize((size_t)s.n + p.halo_slot.size());
    p.pub.resize((size_t)s.n);
    p.orig.resize((size_t)s.n);
    for_parts(s.parts, s.n, [&](int32_t q, uint32_t *remote) {
        const TilePart &pt = p.parts[(size_t)q];
        const std::vector<int32_t> &own = p.own[(size_t)q], &halo = p.halo[(size_t)q];
        for (int32_t h = 0; h < pt.n_halo; ++h) {
            const int32_t g = halo[(size_t)h];
            remote[g] = (uint32_t)(pt.n_own + h);
            p.site[(size_t)(pt.site_begin + pt.n_own + h)] = s.site_off + g;
            p.halo_slot[(size_t)(pt.halo_begin + h)] = p.parts[(size_t)p.part[(size_t)g]].word_begin + p.word[(size_t)g];
        }
        int c = 0;
        uint32_t code = 0;
        for (int32_t k = 0; k < pt.n_own; ++k) {
            while (k >= p.classes[(size_t)q * a.n_colours + c].end) ++c;
            const int32_t g = own[(size_t)k], w0 = p.word[(size_t)g];
            p.site[(size_t)(pt.site_begin + k)] = s.site_off + g;
            p.orig[(size_t)(pt.own_begin + k)] = s.orig[g];
            p.pub[(size_t)(pt.own_begin + k)] = w0 < 0 ? -1 : pt.word_begin + w0;
            const size_t at = (size_t)(pt.own_begin + k) * W;
            const int64_t e0 = s.row_ptr[g], deg = s.row_ptr[g + 1] - e0;
            for (int w = 0; w < W; ++w) {
                uint32_t link = (uint32_t)k;
                float J = 0.0f;
                if (w < deg) {
                    const int32_t j = s.col[e0 + w];
                    link = (p.part[(size_t)j] == q ? (uint32_t)p.local[(size_t)j] : remote[j]) | (j < s.cstart[c] ? 0x10000u : 0u);
                    J = (float)s.J[e0 + w];
                }
                if (a.n_codes) {
                    code = exchange_code(p.codes, J, code);
                    ((uint32_t *)p.rows.get())[at + w] = link | code << 17;
                } else {
                    int2 x = make_int2((int)link, 0);
                    std::memcpy(&x.y, &J, sizeof J);
                    ((int2 *)p.rows.get())[at + w] = x;
                }
            }
        }
    });
}

// Byte offsets of the block's shared memory; returns the bytes needed.
size_t tile_layout(TileArgs &a, const TilePlan &p, int threads) {
    auto align = [](size_t x) { return (x + 15) / 16 * 16; };
    a.cap = (p.max_loc + 1) & ~1;
    size_t at = align((size_t)a.cap * 12);
    a.rows_off = (int32_t)at;
    if (a.mem >= 2) at = align(at + (size_t)p.max_own * a.width * (a.n_codes ? 4 : 8));
    a.orig_off = (int32_t)at;
    if (a.mem >= 1) at = align(at + (size_t)p.max_own * 4);
    a.pub_off = (int32_t)at;
    if (a.mem >= 1) at = align(at + (size_t)p.max_own * 4);
    a.slot_off = (int32_t)at;
    if (a.mem >= 1) at = align(at + (size_t)p.max_halo * 4);
    a.code_off = (int32_t)at;
    at = align(at + (size_t)a.n_codes * sizeof(float));
    a.cls_off = (int32_t)at;
    at = align(at + (size_t)a.n_colours * sizeof(TileClass));
    a.part_off = (int32_t)at;
    if (a.mem == 0) return at + (size_t)(threads / 32) * (4 * sizeof(double) + sizeof(uint32_t));
    return at + (size_t)(1 + a.two_buffers) * threads * 5 * sizeof(float);
}

}  // namespace

void tile_tables(const TileArgs &a, const TileShape &s, TilePlan &p) { write_tables(a, s, p); }

// Raises the kernel's shared-memory limit to the device's (not to this plan's size: the limit
// belongs to the kernel, which other contexts launch too).
int tile_shape(TileArgs &a, const TileShape &s, TilePlan &p, size_t *smem) {
    int dev = 0, most = 0;
    if (cudaGetDevice(&dev) != cudaSuccess ||
        cudaDeviceGetAttribute(&most, cudaDevAttrMaxSharedMemoryPerBlockOptin, dev) != cudaSuccess)
        return 0;
    int own = 1, halo = 0;  // widest class of a part, remote words of one
    for (const TileClass &cl : p.classes) {
        own = std::max(own, cl.end - cl.begin);
        halo = std::max(halo, cl.halo_end - cl.halo_begin);
    }
    // equal rounds over the widest class, and its remote words in one round of two per thread
    // where that many threads fit; below the largest, a warp more costs less than a round
    const int rounds = (own + kTileThreads - 1) / kTileThreads;
    const int best = std::min(kTileThreads, std::max({64, ((own + rounds - 1) / rounds + 31) / 32 * 32, (halo / 2 + 31) / 32 * 32}));
    cudaFuncAttributes rec;  // loads the record kernel now, not in the first (timed) launch
    if (cudaFuncGetAttributes(&rec, tile_record_kernel) != cudaSuccess) return 0;
    exchange_values(s.J, s.row_ptr[s.n], p.codes);
    const bool words = p.codes.size() <= (size_t)kTileCodes && !a.pass.pol32 && !a.cubic;
    // pairs in shared memory, then words there, then words (or pairs) through L1
    int found = 0;
    for (int form = 0; form < 4 && !found; ++form) {
        if (form == 1 && !words) continue;
        a.mem = form == 0 ? 2 : 3 - form;
        a.n_codes = form > 0 && words ? (int32_t)p.codes.size() : 0;
        a.two_buffers = a.mem > 0 ? 1 : 0;  // alone, one buffer: it is long empty when a large part ends its MCS
        const TileFn f = select_tile(a);
        cudaFuncAttributes fa;
        if (cudaFuncGetAttributes(&fa, f) != cudaSuccess ||
            cudaFuncSetAttribute(f, cudaFuncAttributeMaxDynamicSharedMemorySize, most - (int)fa.sharedSizeBytes) != cudaSuccess)
            return 0;
        // the last form gives up threads for spins (at least half of them)
        for (int nt = best; nt >= (a.mem == 0 ? std::min(best, kTileThreads / 2) : best) && !found; nt -= 32) {
            *smem = tile_layout(a, p, nt);
            int nb = 0;
            if (*smem + fa.sharedSizeBytes > (size_t)most) continue;
            if (cudaOccupancyMaxActiveBlocksPerMultiprocessor(&nb, f, nt + kTileRecord, *smem) != cudaSuccess || nb < 1) continue;
            found = nt;
        }
    }
    if (!found) return 0;
    p.columns = p.columns && own <= found;
    for (int32_t q = 0; q < s.parts; ++q) {  // a thread's FP32 sums: at most kTileRun attempts
        int32_t run = 0;
        for (int c = 0; c < a.n_colours; ++c) {
            const TileClass &cl = p.classes[(size_t)q * a.n_colours + c];
            run += (cl.end - cl.begin + found - 1) / found;
        }
        if (run > kTileRun) return 0;
        p.run = std::max(p.run, run);
    }
    write_tables(a, s, p);
    return found;
}

int launch_tile(const TileArgs &a, int threads, size_t smem, void *stream) {
    cudaStream_t st = (cudaStream_t)stream;
    // no word may carry a tag of this launch before it is stored (the MCS counter can be set back)
    cudaError_t e = cudaMemsetAsync(a.mail, 0, ((size_t)a.n_mail << a.pass.log2R) * sizeof(float4), st);
    if (e != cudaSuccess) return (int)e;
    cudaLaunchConfig_t cfg = {};
    cfg.gridDim = dim3((unsigned)(a.P << a.pass.log2R));
    cfg.blockDim = dim3((unsigned)(threads + kTileRecord));
    cfg.dynamicSmemBytes = smem;
    cfg.stream = st;
    cudaLaunchAttribute attr[1];
    attr[0].id = cudaLaunchAttributeCooperative;
    attr[0].val.cooperative = 1;
    cfg.attrs = attr;
    cfg.numAttrs = 1;
    if ((e = cudaLaunchKernelEx(&cfg, select_tile(a), a)) != cudaSuccess) return (int)e;
    return launch_tile_record(a, stream);
}

int launch_tile_record(const TileArgs &a, void *stream) {
    const int64_t warps = (int64_t)a.mcs << a.pass.log2R;
    tile_record_kernel<<<(unsigned)((warps + 3) / 4), 128, 0, (cudaStream_t)stream>>>(a);
    return (int)cudaGetLastError();
}

}  // namespace vegas
