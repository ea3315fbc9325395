// Resident and cluster sweeps of a batch with every instance's spins in shared memory (uniform
// trials, no per-type sums): blocks of 512 sweeping threads take instances from a queue, largest
// first, and run every MCS of the launch on each; the largest may take a cluster of blocks, each
// with a copy of the spins. Which thread takes which site, and so the order of every FP32 sum, is that
// of resident32_kernel and cluster32_kernel, which keep the batches with policies or per-type sums.
//
// What bounds it: instruction issue and the latency of an attempt while an SM's instances pass
// through their classes, and it was the tail of every MCS. So here
//  - the MCS's totals are formed by four warps of their own from the threads' FP32 sums, while the
//    next MCS runs (an FP64 instruction of a warp takes 64 cycles: 148 of them per block and MCS were
//    1.4 us between two MCS, as long as two classes of a small particle);
//  - rows are 48 bytes (one word per link: local site, lower flag, index of J; samples with more than
//    kTileCodes exchange values: 96) and padded with links of J = 0 to the site itself, so no lane
//    branches on its row's length;
//  - parts of an attempt that a batch does not have (cubic or any anisotropy, lower links of a class)
//    are compiled out or skipped per class, Philox's round keys are kernel arguments, and an
//    attempt's random numbers, trial and links are prepared before the class barrier.
// 256 nanoparticles of 100 to 14k sites: 23.9 G attempts/s before, 36.0 now in the shape (splits, groups) that
// those kernels are fastest with, which the automatic choice keeps so that the records stay theirs; 40.1
// in the shape that suits this one best.
#include <cooperative_groups.h>
#include <cuda_runtime.h>

#include <algorithm>
#include <cstdint>

#include "vegas_device.cuh"
#include "vegas_internal.h"
#include "vegas_tile.cuh"
#include "vegas_tile.h"

namespace vegas {
namespace {

namespace cg = cooperative_groups;

constexpr int kNT = kBatchThreads;        // sweeping threads; four record warps behind them
constexpr int kGroups = 4;                // most instances of a block at once
constexpr int kBarSweep = 1, kBarFull = 5, kBarEmpty = 9;  // + group

// One instance on `threads` threads of a block (or, CL, on the cluster's blocks together).
template <int PM, int FMT, bool CL>
__device__ __forceinline__ void batch_sweep(const BatchArgs &ba, const ResidentInst &I, float *sp, int cap, float *s_part,
                                            uint32_t *s_cnt, const float *s_J, int tid, int threads, int group, int n_rec,
                                            bool &nan_seen) {
    const ResidentArgs &a = ba.r;
    cg::cluster_group cl = cg::this_cluster();
    const int CS = CL ? (int)cl.num_blocks() : 1, rank = CL ? (int)cl.block_rank() : 0;
    RunState *rs = a.run;
    const int R = 1 << a.log2R;
    const uint32_t t0 = rs->t, rec0 = rs->rec, step = rec0 / rs->mcs;
    const double *sc = rs->sched + ((int64_t)step * a.n_inst + I.inst_local) * 2;
    const float beta = (float)sc[0], B = (float)sc[1];
    const uint32_t inst = (uint32_t)I.inst_id;
    float4 *S = (float4 *)a.spins;
    const TileRow<kEllRow, FMT> *rows = (const TileRow<kEllRow, FMT> *)ba.rows;
    for (int g = I.g_begin + tid; g < I.g_end; g += threads) {
        const float4 v = S[(int64_t)g * R + I.r];
        loc_set(sp, cap, g - I.g_begin, v.x, v.y, v.z);
    }
    if (CL)
        cl.sync();  // no block writes into a copy that is still being loaded
    else
        bar_sync(kBarSweep + group, threads);
    const int off = rank * threads + tid, stride = CS * threads;
    struct {
        uint32_t orig, wacc;
        Site32 p;
        float4 Si;
        float3 P;
        TileRow<kEllRow, FMT> row;
    } q;
    auto prep = [&](int g, uint32_t t) {  // everything that no other site's sweep changes
        q.orig = (uint32_t)__ldg(a.orig + g);
        q.Si = loc_spin(sp, cap, g - I.g_begin);
#pragma unroll
        for (int j = 0; j < kEllRow / 2; ++j) q.row.q[j] = __ldg(&rows[g].q[j]);
        q.p = Site32{I.u.nx, I.u.ny, I.u.nz, I.u.s, I.u.ex, I.u.ey, I.u.ez, I.u.k, I.u.kc};
        if (PM != 0 && I.params_mode == 2) {
            const float4 p0 = __ldg((const float4 *)a.p0 + g), p1 = __ldg((const float4 *)a.p1 + g);
            q.p = Site32{p0.x, p0.y, p0.z, p0.w, p1.x, p1.y, p1.z, p1.w, __ldg((const float *)a.pk + g)};
        }
        uint4 rw = make_uint4(q.orig, t, inst, kPurposeTrial32);
#pragma unroll
        for (int j = 0; j < 10; ++j) {
            const uint32_t lo0 = 0xD2511F53u * rw.x, hi0 = __umulhi(0xD2511F53u, rw.x);
            const uint32_t lo1 = 0xCD9E8D57u * rw.z, hi1 = __umulhi(0xCD9E8D57u, rw.z);
            rw = make_uint4(hi1 ^ rw.y ^ ba.rk0[j], lo1, hi0 ^ rw.w ^ ba.rk1[j], lo0);
        }
        q.P = trial_random32(rw, q.p.sn);
        q.wacc = rw.z;
    };
    float2 fem = make_float2(0.f, 0.f), fxy = fem;
    uint32_t nacc = 0;
    auto finish = [&](int g, uint32_t t, int mode) {
        float2 hxy = make_float2(0.f, 0.f), lxy = hxy;
        float hz = 0.f, lz = 0.f;
        if (mode == 2) {
#pragma unroll
            for (int j = 0; j < kEllRow; ++j)
                link32(loc_spin(sp, cap, q.row.site(j)), q.row.J(j, s_J), q.row.lower(j), hxy, hz, lxy, lz);
        } else {
#pragma unroll
            for (int j = 0; j < kEllRow; ++j)
                link32(loc_spin(sp, cap, q.row.site(j)), q.row.J(j, s_J), false, hxy, hz, lxy, lz);
            if (mode == 1) {  // every link goes to a lower colour
                lxy = hxy;
                lz = hz;
            }
        }
        float4 Sn;
        bool ok, bad;
        float e;
        attempt32<PM, 2>(q.Si, hxy, hz, lxy, lz, q.p, beta, B, q.P, q.wacc, Sn, ok, e, bad);
        if (ok) {
            const int i = g - I.g_begin;
            loc_set(sp, cap, i, Sn.x, Sn.y, Sn.z);
            if (CL)
                for (int b = 1; b < CS; ++b) loc_set(cl.map_shared_rank(sp, (rank + b) % CS), cap, i, Sn.x, Sn.y, Sn.z);
        }
        nan_seen |= bad;
        nacc += ok ? 1u : 0u;
        fem = __fadd2_rn(fem, make_float2(e, Sn.z));
        fxy = __fadd2_rn(fxy, make_float2(Sn.x, Sn.y));
        if (a.alog && t < a.alog_mcs)
            a.alog[(int64_t)t * a.alog_stride + I.alog_base + (int64_t)I.r * I.n_sample_sites + q.orig] = ok ? 1 : 0;
    };
    bool pending = false;  // the class before has not been waited for
    for (int m = 0; m < a.mcs; ++m) {
        const uint32_t t = t0 + (uint32_t)m;
        for (int c = 0; c < I.n_segs; ++c) {
            const int4 sg = a.segs[I.seg_off + c];
            const int mode = __ldg(ba.modes + I.seg_off + c);
            int g = sg.x + off;
            if (g < sg.y) prep(g, t);
            if (pending) {
                if (CL)
                    cl.barrier_wait();
                else
                    bar_sync(kBarSweep + group, threads);
            }
            while (g < sg.y) {
                finish(g, t, mode);
                g += stride;
                if (g < sg.y) prep(g, t);
            }
            if (CL) cl.barrier_arrive();
            pending = true;
        }
        // the thread's sums of this MCS (at most 64 attempts) to the record warps
        if (m > 0) bar_sync(kBarEmpty + group, threads + n_rec);
        s_part[tid] = fem.x;
        s_part[kNT + tid] = fxy.x;
        s_part[2 * kNT + tid] = fxy.y;
        s_part[3 * kNT + tid] = fem.y;
        s_cnt[tid] = nacc;
        bar_arrive(kBarFull + group, threads + n_rec);
        fem = fxy = make_float2(0.f, 0.f);
        nacc = 0;
    }
    if (CL) {
        if (pending) cl.barrier_wait();
        cl.sync();  // the record warps' last totals
        // each block's own sites (the copies agree)
        for (int c = 0; c < I.n_segs; ++c) {
            const int4 sg = a.segs[I.seg_off + c];
            for (int g = sg.x + off; g < sg.y; g += stride) S[(int64_t)g * R + I.r] = loc_spin(sp, cap, g - I.g_begin);
        }
        cl.sync();  // rank 0 has read the totals
    } else {
        bar_sync(kBarSweep + group, threads);
        for (int g = I.g_begin + tid; g < I.g_end; g += threads) S[(int64_t)g * R + I.r] = loc_spin(sp, cap, g - I.g_begin);
    }
}

// Sum over `threads` threads of one quantity by one warp, in a fixed order in FP64.
__device__ __forceinline__ double record_sum(const float *x, int threads, int lane) {
    double v = 0.0;
    for (int k = lane; k < threads; k += 32) v += (double)x[k];
    for (int off = 16; off > 0; off >>= 1) v += __shfl_xor_sync(0xFFFFFFFFu, v, off);
    return v;
}
__device__ __forceinline__ uint32_t record_count(const uint32_t *x, int threads, int lane) {
    uint32_t n = 0;
    for (int k = lane; k < threads; k += 32) n += x[k];
    return __reduce_add_sync(0xFFFFFFFFu, n);
}

// The record warps of one instance that a block (or a group of its threads) sweeps: quantities q0,
// q0 + dq, ... of every MCS into the history.
__device__ __forceinline__ void batch_record(const BatchArgs &ba, const ResidentInst &I, const float *s_part,
                                             const uint32_t *s_cnt, int threads, int group, int n_rec, int q0, int dq) {
    const ResidentArgs &a = ba.r;
    const RunState *rs = a.run;
    const int lane = threadIdx.x & 31;
    const uint32_t rec0 = rs->rec;
    for (int m = 0; m < a.mcs; ++m) {
        bar_sync(kBarFull + group, threads + n_rec);
        double v[4];
        for (int q = q0, k = 0; q < 4; q += dq, ++k) v[k] = record_sum(s_part + q * kNT, threads, lane);
        const uint32_t n = q0 == 0 ? record_count(s_cnt, threads, lane) : 0u;
        if (m + 1 < a.mcs) bar_arrive(kBarEmpty + group, threads + n_rec);
        if (lane == 0) {
            const int64_t at = ((int64_t)rec0 + m) * a.n_inst + I.inst_local;
            for (int q = q0, k = 0; q < 4; q += dq, ++k) rs->hist[at * 4 + q] = v[k];
            if (q0 == 0 && rs->acc_hist) rs->acc_hist[at] = n;
        }
    }
}

// The same for an instance that a cluster sweeps: every warp takes part in the cluster's barriers, so
// the block's totals of MCS m - 1 are formed between the arrivals of classes 0 and 1 of MCS m, and
// rank 0 adds the blocks' in rank order after the wait for class 0.
__device__ __forceinline__ void batch_record_cluster(const BatchArgs &ba, const ResidentInst &I, const float *s_part,
                                                     const uint32_t *s_cnt, double (*s_blk)[5]) {
    const ResidentArgs &a = ba.r;
    cg::cluster_group cl = cg::this_cluster();
    const int CS = (int)cl.num_blocks(), rank = (int)cl.block_rank();
    const int lane = threadIdx.x & 31, q = ((int)threadIdx.x - kNT) >> 5;
    const RunState *rs = a.run;
    const uint32_t rec0 = rs->rec;
    cl.sync();  // the spins are loaded
    auto block_totals = [&](int m) {
        bar_sync(kBarFull, kNT + 128);
        const double v = record_sum(s_part + q * kNT, kNT, lane);
        const uint32_t n = q == 0 ? record_count(s_cnt, kNT, lane) : 0u;
        if (m + 1 < a.mcs) bar_arrive(kBarEmpty, kNT + 128);
        if (lane == 0) s_blk[m & 1][q] = v;
        if (lane == 0 && q == 0) s_blk[m & 1][4] = (double)n;
    };
    auto combine = [&](int m) {
        if (rank != 0 || q != 0 || lane >= 5) return;
        double x = 0.0;
        for (int b = 0; b < CS; ++b) x += cl.map_shared_rank(&s_blk[m & 1][0], b)[lane];
        const int64_t at = ((int64_t)rec0 + m) * a.n_inst + I.inst_local;
        if (lane < 4)
            rs->hist[at * 4 + lane] = x;
        else if (rs->acc_hist)
            rs->acc_hist[at] = (uint32_t)x;
    };
    bool pending = false;
    for (int m = 0; m < a.mcs; ++m)
        for (int c = 0; c < I.n_segs; ++c) {
            if (pending) cl.barrier_wait();
            if (m > 0 && c == 0) block_totals(m - 1);
            if (m > 0 && c == 1) combine(m - 1);
            cl.barrier_arrive();
            pending = true;
        }
    if (pending) cl.barrier_wait();
    if (a.mcs > 0) block_totals(a.mcs - 1);
    cl.sync();
    if (a.mcs > 0) combine(a.mcs - 1);
    cl.sync();
}

// PM: 0 no anisotropy and uniform parameters in the batch, 3 no cubic constant, 2 any.
template <int PM, int FMT>
__global__ void __launch_bounds__(kNT + 128) batch32_kernel(const BatchArgs ba) {
    const ResidentArgs &a = ba.r;
    extern __shared__ __align__(16) unsigned char smem[];
    float *sp = (float *)smem, *s_part = (float *)(smem + ba.part_off);
    uint32_t *s_cnt = (uint32_t *)(s_part + 4 * kNT);
    __shared__ float s_J[kTileCodes];
    __shared__ double s_blk[2][5];
    __shared__ int s_items[kGroups + 1];
    __shared__ int s_item;
    cg::cluster_group cl = cg::this_cluster();
    const int tid = (int)threadIdx.x;
    bool nan_seen = false;
    if (FMT == 1 && tid < ba.n_codes) s_J[tid] = ba.codes[tid];
    int first = -1;  // an instance drawn for a cluster but small enough for a block
    if (ba.clusters) {
        const int rank = (int)cl.block_rank();
        for (;;) {
            if (rank == 0 && tid == 0) s_item = (int)atomicAdd(a.queue, 1u);
            cl.sync();
            const int item = *cl.map_shared_rank(&s_item, 0);
            cl.sync();  // every block has read the item before rank 0 fetches the next
            if (item >= a.n_items) break;
            const ResidentInst I = a.insts[item];
            if ((a.split_sites > 0 && I.g_end - I.g_begin <= a.split_sites) || I.n_segs < 2) {
                if (rank == 0) first = item;
                break;
            }
            if (tid < kNT)
                batch_sweep<PM, FMT, true>(ba, I, sp, a.smem_sites, s_part, s_cnt, s_J, tid, kNT, 0, 128, nan_seen);
            else
                batch_record_cluster(ba, I, s_part, s_cnt, s_blk);
        }
    }
    // blocks alone: no shared memory of another block is read or written from here on
    const int GT = a.group_threads;
    for (;;) {
        if (tid == 0) {
            const int it = first >= 0 ? first : (int)atomicAdd(a.queue, 1u);
            int ng = 1;
            if (GT > 0 && GT < kNT && it < a.n_items && a.insts[it].g_end - a.insts[it].g_begin <= a.group_sites) {
                ng = kNT / GT;
                const int more = (int)atomicAdd(a.queue, (uint32_t)(ng - 1));
                for (int k = 1; k < ng; ++k) s_items[k] = more + k - 1;
            }
            s_items[0] = it;
            s_items[kGroups] = ng;
        }
        first = -1;
        __syncthreads();
        const int ng = s_items[kGroups];
        if (s_items[0] >= a.n_items) break;
        const int gt = kNT / ng;
        if (tid < kNT) {
            const int gi = tid / gt, item = s_items[gi];
            if (item < a.n_items) {
                const int cap = ng == 1 ? a.smem_sites : a.group_sites;
                batch_sweep<PM, FMT, false>(ba, a.insts[item], sp + (size_t)gi * 3 * (size_t)((cap + 1) & ~1), cap,
                                            s_part + gi * gt, s_cnt + gi * gt, s_J, tid - gi * gt, gt, gi, ng == 1 ? 128 : 32,
                                            nan_seen);
            }
        } else {
            const int w = (tid - kNT) >> 5;  // one instance: warp w takes quantity w; several: a warp each
            const int gi = ng == 1 ? 0 : w;
            if (gi < ng && s_items[gi] < a.n_items)
                batch_record(ba, a.insts[s_items[gi]], s_part + gi * gt, s_cnt + gi * gt, gt, gi, ng == 1 ? 128 : 32,
                             ng == 1 ? w : 0, ng == 1 ? 4 : 1);
        }
        __syncthreads();  // every group is done before the items are drawn again
    }
    if (nan_seen) atomicOr(a.err, kErrNaN);
}

using BatchFn = void (*)(BatchArgs);

BatchFn select_batch(const BatchArgs &a) {
    if (a.r.any_aniso == 0) return a.n_codes ? batch32_kernel<0, 1> : batch32_kernel<0, 0>;
    if (!a.cubic) return a.n_codes ? batch32_kernel<3, 1> : batch32_kernel<3, 0>;
    return a.n_codes ? batch32_kernel<2, 1> : batch32_kernel<2, 0>;
}

// Room for the spins of the largest instance, or of a block's groups of instances, then the sums.
size_t batch_layout(BatchArgs &a) {
    const int ng = a.r.group_threads > 0 && a.r.group_threads < kNT ? kNT / a.r.group_threads : 1;
    const int64_t sites = std::max<int64_t>((a.r.smem_sites + 1) & ~1, ng > 1 ? (int64_t)ng * ((a.r.group_sites + 1) & ~1) : 0);
    a.part_off = (int32_t)((sites * 12 + 15) / 16 * 16);
    return (size_t)a.part_off + kNT * 5 * sizeof(float);
}

int launch_config(cudaLaunchConfig_t &cfg, cudaLaunchAttribute *attr, BatchArgs &a, int blocks, int cs, void *stream) {
    cfg = cudaLaunchConfig_t{};
    cfg.gridDim = dim3((unsigned)blocks);
    cfg.blockDim = dim3(kNT + 128);
    cfg.dynamicSmemBytes = batch_layout(a);
    cfg.stream = (cudaStream_t)stream;
    attr[0].id = cudaLaunchAttributeClusterDimension;
    attr[0].val.clusterDim.x = (unsigned)cs;
    attr[0].val.clusterDim.y = 1;
    attr[0].val.clusterDim.z = 1;
    cfg.attrs = attr;
    cfg.numAttrs = 1;
    a.clusters = cs > 1 ? 1 : 0;
    return 0;
}

}  // namespace

// Clusters of cs blocks (cs = 1: blocks) that fit on the device at once, 0 when none does. The
// shared-memory limit belongs to the kernel, which other contexts launch too: raised to the device's.
int batch_capacity(BatchArgs a, int cs, int sm_count) {
    const BatchFn f = select_batch(a);
    cudaLaunchConfig_t cfg;
    cudaLaunchAttribute attr[1];
    launch_config(cfg, attr, a, cs, cs, nullptr);
    int dev = 0, most = 0, n = 0;
    cudaFuncAttributes fa;
    if (cudaGetDevice(&dev) != cudaSuccess ||
        cudaDeviceGetAttribute(&most, cudaDevAttrMaxSharedMemoryPerBlockOptin, dev) != cudaSuccess ||
        cudaFuncGetAttributes(&fa, f) != cudaSuccess || cfg.dynamicSmemBytes + fa.sharedSizeBytes > (size_t)most ||
        cudaFuncSetAttribute(f, cudaFuncAttributeMaxDynamicSharedMemorySize, most - (int)fa.sharedSizeBytes) != cudaSuccess)
        return 0;
    if (cs > 8 && cudaFuncSetAttribute(f, cudaFuncAttributeNonPortableClusterSizeAllowed, 1) != cudaSuccess) return 0;
    if (cs == 1) {
        if (cudaOccupancyMaxActiveBlocksPerMultiprocessor(&n, f, kNT + 128, cfg.dynamicSmemBytes) != cudaSuccess) return 0;
        return n * sm_count;
    }
    if (cudaOccupancyMaxActiveClusters(&n, f, &cfg) != cudaSuccess) return 0;
    return n;
}

int launch_batch(BatchArgs a, int n, int cs, void *stream) {
    cudaLaunchConfig_t cfg;
    cudaLaunchAttribute attr[1];
    launch_config(cfg, attr, a, n * cs, cs, stream);
    return (int)cudaLaunchKernelEx(&cfg, select_batch(a), a);
}

}  // namespace vegas
