// Device pieces of the sweeps with spins in shared memory: named barriers, mailbox words, spins and
// rows of links.
#pragma once

#include <cuda_runtime.h>

#include <cstdint>

#include "vegas_internal.h"

namespace vegas {
namespace {

__device__ __forceinline__ void bar_sync(int id, int n) { asm volatile("bar.sync %0, %1;" ::"r"(id), "r"(n) : "memory"); }
__device__ __forceinline__ void bar_arrive(int id, int n) {
    asm volatile("bar.arrive %0, %1;" ::"r"(id), "r"(n) : "memory");
}

// A mailbox word in one 128-bit access (single-copy atomic), through L2.
__device__ __forceinline__ void mail_store(float4 *p, float x, float y, float z, uint32_t tag) {
    const uint64_t lo = (uint64_t)__float_as_uint(x) | (uint64_t)__float_as_uint(y) << 32;
    const uint64_t hi = (uint64_t)__float_as_uint(z) | (uint64_t)tag << 32;
    asm volatile("{\n\t.reg .b128 q;\n\tmov.b128 q, {%1, %2};\n\tst.relaxed.gpu.global.b128 [%0], q;\n\t}" ::"l"(p), "l"(lo),
                 "l"(hi)
                 : "memory");
}
__device__ __forceinline__ float4 mail_load(const float4 *p) {
    uint64_t lo, hi;
    asm volatile("{\n\t.reg .b128 q;\n\tld.relaxed.gpu.global.b128 q, [%2];\n\tmov.b128 {%0, %1}, q;\n\t}"
                 : "=l"(lo), "=l"(hi)
                 : "l"(p)
                 : "memory");
    return make_float4(__uint_as_float((uint32_t)lo), __uint_as_float((uint32_t)(lo >> 32)), __uint_as_float((uint32_t)hi),
                       __uint_as_float((uint32_t)(hi >> 32)));
}

// The barrier and the logical and of every thread's ok.
__device__ __forceinline__ bool bar_and(int id, int n, bool ok) {
    int all;
    asm volatile("{\n\t.reg .pred p, q;\n\tsetp.ne.s32 p, %1, 0;\n\tbar.red.and.pred q, %2, %3, p;\n\tselp.s32 %0, 1, 0, q;\n\t}"
                 : "=r"(all)
                 : "r"((int)ok), "r"(id), "r"(n)
                 : "memory");
    return all != 0;
}

__device__ __forceinline__ uint64_t tile_ns() {
    uint64_t t;
    asm volatile("mov.u64 %0, %%globaltimer;" : "=l"(t));
    return t;
}

// The spin of local site i: x and y as one 8-byte pair, z in an array of its own (two loads).
__device__ __forceinline__ float4 loc_spin(const float *sp, int cap, int i) {
    const float2 xy = ((const float2 *)sp)[i];
    return make_float4(xy.x, xy.y, sp[2 * cap + i], 0.f);
}
__device__ __forceinline__ void loc_set(float *sp, int cap, int i, float x, float y, float z) {
    ((float2 *)sp)[i] = make_float2(x, y);
    sp[2 * cap + i] = z;
}

// A fixed row of W links: (local site | lower flag << 16, J) pairs, or with FMT 1 one word per link,
// the pair's first word with J's index in the sample's table of exchange values from bit 17 on.
template <int W, int FMT>
struct TileRow {
    int4 q[W / 2];
    __device__ __forceinline__ int site(int j) const { return (j & 1 ? q[j / 2].z : q[j / 2].x) & 0xFFFF; }
    __device__ __forceinline__ bool lower(int j) const { return ((j & 1 ? q[j / 2].z : q[j / 2].x) >> 16) != 0; }
    __device__ __forceinline__ float J(int j, const float *) const { return __int_as_float(j & 1 ? q[j / 2].w : q[j / 2].y); }
};
template <int W>
struct TileRow<W, 1> {
    int2 q[W / 2];
    __device__ __forceinline__ int site(int j) const { return (j & 1 ? q[j / 2].y : q[j / 2].x) & 0xFFFF; }
    __device__ __forceinline__ bool lower(int j) const { return ((j & 1 ? q[j / 2].y : q[j / 2].x) & 0x10000) != 0; }
    __device__ __forceinline__ float J(int j, const float *t) const { return t[(j & 1 ? q[j / 2].y : q[j / 2].x) >> 17]; }
};

}  // namespace
}  // namespace vegas
