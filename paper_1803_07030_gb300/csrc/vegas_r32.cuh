// The replica-batched FP32 colour pass (R = 32, rows of six links): shared by the translation
// unit of the staged kernels (no policy table, or a table read per site) and the one of the
// kernels specialised to a single update policy.
#pragma once

#include <cuda_runtime.h>

#include <cstdint>

#include "vegas_device.cuh"
#include "vegas_internal.h"
#include "vegas_staged.cuh"

namespace vegas {
namespace {

// Replica-batched sweep (R = 32): one warp = one site x 32 replicas, depth-2 pipeline. A
// warp takes blocks of eight consecutive sites from the pass's ticket counter, so the blocks
// in flight stay about one per warp and consecutive in memory order however unevenly the
// warps progress: the neighbour rows they share are still in L2 when the last of them reads
// them. The eight groups of a block are unrolled, so every ring slot and offset is a
// constant: group j of a block computes from row slot j & 1 and its link slot; the next
// ticket is drawn at j = 0 and its block's links copied at j = 4; rows of group j + 2 (the
// next block's first two at j = 6, 7) are copied at the end of group j.
// POL = 1 adds the sites' update policies (8 bytes each, staged with the caller ids); POL =
// 2 + c does the same for a pass whose sites all have policy c, with the trial of that policy
// alone compiled in (each site's parameter still comes from its entry).
// Rows are kept in planes (384 bytes of a site's 512): what the kernel moves most. A site's seven
// rows come as 168 16-byte pieces, lane + 32 i the i-th of a lane. Per launch on 128^3 sites x 32,
// against rows of 32 float4: 1.21 GB of DRAM traffic against 1.48, 205 M warp instructions
// against 212, issue 67% against 62, 253 us against 282 (under ncu); on 256^3 1.90 ms against 2.04.
// Issue, the shared-memory pipe (61%) and DRAM (60%) are now about equally busy. The Philox round keys
// are kernel arguments, which frees 20 registers; yet 24 warps per SM (8 x 3) stay the best:
// 513 us per MCS on 128^3, 28 warps 522, 32 warps 544, 36 warps 567, 16 warps 567. Also tried:
// alternate directions of the passes, so that one starts where the other ended in L2 (no
// change), a finer cut of the last round of blocks (none), the loop over a block unrolled by two
// (544) and four (521). The block's partial sums are formed in each warp's own shared-memory
// area once its sweep is done, so the block needs no other shared memory.
template <int POL>
struct R32Shape {
    static constexpr int DEG = 6, D = 2, BS = 8;
    static constexpr int WARPS = 8, MIN_BLOCKS = 3;
    static constexpr int ROW = kPlanarRow * 4;  // bytes
    static constexpr int ROWS = D * (DEG + 1) * ROW;
    static constexpr int LINK_BYTES = BS * DEG * 8;
    static constexpr int POL_OFF = LINK_BYTES + BS * 4;
    static constexpr int SLOT = POL_OFF + (POL ? BS * 8 : 0);
    static constexpr int WARP_BYTES = ROWS + 2 * SLOT;
};

// Fixed-order block sums of (E, Mx, My, Mz) per replica and the accepted counts, through the
// warps' own areas of the dynamic shared memory (the same order as block_partials: a butterfly
// inside the warp, then the warps in order).
__device__ __forceinline__ void block_partials_r32(double v[4], uint32_t nacc, unsigned char *smem, int warp_bytes,
                                                   double *out, uint32_t *acc) {
    const int lane = threadIdx.x & 31, warp = threadIdx.x >> 5;
    double *mine = (double *)(smem + (size_t)warp * warp_bytes);
#pragma unroll
    for (int q = 0; q < 4; ++q) mine[lane * 4 + q] = v[q];
    ((uint32_t *)(mine + 32 * 4))[lane] = nacc;
    __syncthreads();
    if (threadIdx.x < 32) {
        double a4[4] = {0.0, 0.0, 0.0, 0.0};
        uint32_t na = 0;
        for (int w = 0; w < (int)(blockDim.x >> 5); ++w) {
            const double *o = (const double *)(smem + (size_t)w * warp_bytes);
#pragma unroll
            for (int q = 0; q < 4; ++q) a4[q] += o[threadIdx.x * 4 + q];
            na += ((const uint32_t *)(o + 32 * 4))[threadIdx.x];
        }
#pragma unroll
        for (int q = 0; q < 4; ++q) out[threadIdx.x * 4 + q] = a4[q];
        if (acc && na) atomicAdd(acc + threadIdx.x, na);
    }
}

__device__ __forceinline__ uint32_t atom_add_acq_rel(uint32_t *p, uint32_t v) {
    uint32_t old;
    asm volatile("atom.acq_rel.gpu.global.add.u32 %0, [%1], %2;" : "=r"(old) : "l"(p), "r"(v) : "memory");
    return old;
}

// Renormalise class-0 block b (its sites x 32 replicas, lane = replica), four rows in flight.
__device__ __forceinline__ void renorm_block32(const PassArgs &a, float4 *S, int b, int lane) {
    const int g0 = a.fold_c0_begin + b * kFoldBlockSites;
    const int n = min(kFoldBlockSites, a.fold_c0_end - g0);
#pragma unroll
    for (int h = 0; h < kFoldBlockSites; h += 4) {
        float4 v[4];
#pragma unroll
        for (int k = 0; k < 4; ++k)
            if (h + k < n) {
                const float *row = (const float *)(S + (int64_t)(g0 + h + k) * 32);
                const float2 xy = __ldcg((const float2 *)row + lane);
                v[k] = make_float4(xy.x, xy.y, __ldcg(row + 64 + lane), 0.f);
            }
#pragma unroll
        for (int k = 0; k < 4; ++k)
            if (h + k < n)
                planar_set((float *)(S + (int64_t)(g0 + h + k) * 32), lane, renorm_spin32(v[k], __ldg(a.fold_norm + g0 + h + k)));
    }
}

// RN = 1 (the step's last class-1 pass of a two-class sample, POL = 0): every attempt stores
// its spin renormalised, and once a block's eight groups are done the warp counts the block
// finished for each class-0 block it read (one per lane, an acquire-release add after the
// block's copies have landed); the warp whose add completes a class-0 block's count of readers
// renormalises that block. No class-1 block reads it afterwards in this pass and nothing else
// reads spins before the pass ends, so every spin is renormalised after its last use of the
// step: the same values as a renormalisation pass after the sweep.
template <int PM, int LM, int POL, int RN = 0>
__global__ void __launch_bounds__(R32Shape<POL>::WARPS * 32, R32Shape<POL>::MIN_BLOCKS) pass32_r32(const PassArgs a) {
    static_assert(RN == 0 || POL == 0, "the folded renormalisation runs without a policy table");
    using Sh = R32Shape<POL>;
    constexpr int DEG = Sh::DEG, D = Sh::D, BS = Sh::BS, R = 32;
    constexpr int ROWS = Sh::ROWS;
    constexpr int LINK_BYTES = Sh::LINK_BYTES;
    constexpr int POL_OFF = Sh::POL_OFF;
    constexpr int SLOT = Sh::SLOT;
    constexpr int WARP_BYTES = Sh::WARP_BYTES;
    static_assert(BS == kFoldBlockSites && kFoldDeps == 32, "the host's blocks of class sites; one per lane");
    extern __shared__ __align__(16) unsigned char smem[];
    const RunState *rs_ = a.run;
    const uint32_t t = rs_->t;
    const uint32_t step_idx = rs_->rec / rs_->mcs;
    const int lane = threadIdx.x & 31, warp = threadIdx.x >> 5;
    const int r = lane;
    unsigned char *wbase = smem + warp * WARP_BYTES;
    unsigned char *lslots = wbase + ROWS;
    float4 *S = (float4 *)a.spins;
    // a site's rows are 7 x 24 16-byte pieces; piece k = lane + 32 i is part of row k / 24. Rows
    // i and i + 3 of a lane are four apart and their pieces at the same place in the row.
    const int k1 = lane + 32, k2 = lane + 64;
    const unsigned char *src0 = (const unsigned char *)S + lane % 24 * 16, *src1 = (const unsigned char *)S + k1 % 24 * 16,
                        *src2 = (const unsigned char *)S + k2 % 24 * 16;
    const int row0 = lane / 24 * 8, row1 = k1 / 24 * 8, row2 = k2 / 24 * 8;  // of a link, bytes
    const int2 *E = (const int2 *)a.edges;
    const uint32_t inst = (uint32_t)(a.inst0 + r);
    const double *sc = rs_->sched + ((int64_t)step_idx * a.n_inst + a.inst_local0 + r) * 2;
    const float beta = (float)sc[0], B = (float)sc[1];
    const float sigma = (POL && rs_->sigma) ? (float)rs_->sigma[a.inst_local0 + r] : 0.f;
    const int g_end = a.g_end;
    auto issue_links = [&](int sb, int slot) {
        if (sb >= g_end) return;
        const int ns = min(BS, g_end - sb);
        unsigned char *dst = lslots + slot * SLOT;
        const unsigned char *src = (const unsigned char *)(E + a.edge_base + (int64_t)(sb - a.site_off) * DEG);
        VEGAS_CHECK(sb >= a.g_begin && sb + ns <= a.n_sites_total, 11, sb);
        VEGAS_CHECK(a.edge_base + (int64_t)(sb - a.site_off + ns) * DEG <= a.n_edges_total, 12, sb);
        VEGAS_CHECK(((uintptr_t)src & 15) == 0, 13, sb);
        if (lane < ns * (DEG / 2)) cp16(dst + 16 * lane, src + 16 * lane);
        if (lane < ns) cp4(dst + LINK_BYTES + 4 * lane, a.orig + sb + lane);
        if (POL && lane < ns) cp8(dst + POL_OFF + 8 * lane, a.pol32 + sb + lane);
    };
    auto issue_rows = [&](int g, int lslot, int j, int rslot) {
        if (g >= g_end) return;
        const unsigned char *lk = lslots + lslot * SLOT + j * (DEG * 8);
        unsigned char *dst = wbase + rslot * (DEG + 1) * Sh::ROW + lane * 16;
        VEGAS_CHECK(g < a.n_sites_total, 14, g);
        const int j0 = *(const int *)(lk + row0), j1 = *(const int *)(lk + row1), j2 = *(const int *)(lk + row2);
        const int j3 = *(const int *)(lk + row0 + 32);
        const int j4 = lane < 16 ? *(const int *)(lk + 40) : g;
        VEGAS_CHECK(min(min(j0, j1), min(j2, j3)) >= 0 && max(max(j0, j1), max(j2, j3)) < a.n_sites_total && j4 >= 0 && j4 < a.n_sites_total, 15, j0);
        cp16(dst, src0 + (int64_t)j0 * (R * 16));
        cp16(dst + 512, src1 + (int64_t)j1 * (R * 16));
        cp16(dst + 1024, src2 + (int64_t)j2 * (R * 16));
        cp16(dst + 1536, src0 + (int64_t)j3 * (R * 16));
        cp16(dst + 2048, src1 + (int64_t)j4 * (R * 16));
        if (lane < 8) cp16(dst + 2560, src2 + (int64_t)g * (R * 16));
    };

    const uint32_t n_blocks = (uint32_t)(g_end - a.g_begin + BS - 1) / BS;  // a ticket past them ends the warp
    // First block: in a short pass the warp's own index, without the wait for thousands of adds
    // to one word (60 x 60 x 52 sites x 32, three blocks per warp: 85 -> 82.5 us per MCS); a long
    // one draws it, which also keeps the warps out of step (128^3: 513 us, with own indexes 518).
    const uint32_t warps = n_blocks < 8 * gridDim.x * Sh::WARPS ? gridDim.x * Sh::WARPS : 0;
    uint32_t tk = blockIdx.x * Sh::WARPS + warp;
    if (warps == 0 && lane == 0) tk = atomicAdd(a.ticket, 1u);
    int sb = a.g_begin + (int)min(__shfl_sync(0xFFFFFFFFu, tk, 0), n_blocks) * BS;
    issue_links(sb, 0);
    cp_commit();
    cp_wait<0>();
    __syncwarp();
    issue_rows(sb, 0, 0, 0);
    cp_commit();
    issue_rows(sb + 1, 0, 1, 1);
    cp_commit();
    Acc32Runs acc;
    int run = 0;  // blocks in the run of FP32 sums (counted per block: 128^3 505.8 -> 501.6 us per MCS)
    bool nan_seen = false;
    const bool log_accepts = a.alog && t < a.alog_mcs;
    int ls = 0;
    while (sb < g_end) {
        int sb2 = g_end;  // the next block (drawn at j = 0, known from j = 4)
#pragma unroll
        for (int j = 0; j < BS; ++j) {
            cp_wait<D - 1>();
            __syncwarp();
            const int g = sb + j;
            if (g < g_end) {
                const unsigned char *slot = lslots + ls * SLOT;
                const uint32_t orig = ((const uint32_t *)(slot + LINK_BYTES))[j];
                uint4 rw = make_uint4(orig, t, inst, kPurposeTrial32);
#pragma unroll
                for (int q = 0; q < 10; ++q) {  // Philox with the round keys as kernel arguments, by constant index
                    const uint32_t lo0 = 0xD2511F53u * rw.x, hi0 = __umulhi(0xD2511F53u, rw.x);
                    const uint32_t lo1 = 0xCD9E8D57u * rw.z, hi1 = __umulhi(0xCD9E8D57u, rw.z);
                    rw = make_uint4(hi1 ^ rw.y ^ a.rk0[q], lo1, hi0 ^ rw.w ^ a.rk1[q], lo0);
                }
                staged_attempt_rw<DEG, PM, LM, POL, RN != 0>(
                    a, (const int4 *)slot + j * (DEG / 2),
                    PlanarRows{(const float *)(wbase + (j & 1) * (DEG + 1) * Sh::ROW), lane}, orig, g, r, R, t, rw, beta, B, S,
                    acc, nan_seen, log_accepts, (const PolicySite32 *)(slot + POL_OFF) + j, sigma);
            }
            __syncwarp();
            if (j == 0 && lane == 0) tk = atomicAdd(a.ticket, 1u);
            if (j == 4) {
                sb2 = a.g_begin + (int)min(warps + __shfl_sync(0xFFFFFFFFu, tk, 0), n_blocks) * BS;
                issue_links(sb2, ls ^ 1);
            }
            if (j + 2 < BS)
                issue_rows(sb + j + 2, ls, j + 2, j & 1);
            else
                issue_rows(sb2 + j + 2 - BS, ls ^ 1, j + 2 - BS, j & 1);
            cp_commit();
        }
        if (RN) {
            const int dep = a.fold_deps[(int64_t)((sb - a.g_begin) / BS) * kFoldDeps + lane];
            __syncwarp();  // every lane's copies of this block have landed and been read
            const bool last = dep >= 0 && atom_add_acq_rel(a.fold_cnt + dep, 1u) + 1u == (uint32_t)__ldg(a.fold_deg + dep);
            for (uint32_t m = __ballot_sync(0xFFFFFFFFu, last); m; m &= m - 1)
                renorm_block32(a, S, __shfl_sync(0xFFFFFFFFu, dep, __ffs(m) - 1), lane);
        }
        if (++run == 64 / BS) {
            acc.flush();
            run = 0;
        }
        sb = sb2;
        ls ^= 1;
    }
    cp_wait<0>();
    if (nan_seen) atomicOr(a.err, kErrNaN);
    acc.flush();
    __syncwarp();  // every lane's copies have landed and been read: the warp's area is free
    block_partials_r32(acc.d, acc.nacc, smem, WARP_BYTES, a.partial + (int64_t)blockIdx.x * R * 4,
                       acc_counters(rs_, a.inst_local0));
}

}  // namespace

// The R = 32 kernels specialised to one update policy (code 1 .. 6), built in their own
// translation unit.
PassFn select_r32_fixed(int pm, int lm, int code);
// The R = 32 kernel of the step's last class-1 pass with the renormalisation folded in
// (lower mode 1: every link of class 1 goes to class 0), in the same unit.
PassFn select_r32_renorm(int pm);

}  // namespace vegas
