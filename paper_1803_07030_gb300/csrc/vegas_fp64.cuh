// FP64 pieces of an attempt shared by the FP64 sweeps: explicit roundings, the uniforms, the sphere
// sampler and the decision.
#pragma once

#include <cuda_runtime.h>

#include <cstdint>

#include "vegas_device.cuh"
#include "vegas_internal.h"

namespace vegas {
namespace {

// ------------------------------------------------------------------ FP64 helpers
// Explicit round-to-nearest operations: the compiler may not fuse them, which keeps the
// FP64 path identical to the CPU oracle built without contraction.
__device__ __forceinline__ double dm(double a, double b) { return __dmul_rn(a, b); }
__device__ __forceinline__ double da(double a, double b) { return __dadd_rn(a, b); }
__device__ __forceinline__ double ds(double a, double b) { return __dsub_rn(a, b); }

// Uniform in [0, 1) with 53 bits: (hi * 2^21 + (lo >> 11)) * 2^-53 (exact).
__device__ __forceinline__ double u53(uint32_t hi, uint32_t lo) {
    const unsigned long long m = ((unsigned long long)hi << 21) | (unsigned long long)(lo >> 11);
    return __dmul_rn(__ull2double_rn(m), 0x1p-53);
}

// 2 m 2^-53 - 1 for m < 2^53: the value the oracle's ds(dm(2.0, u53), 1.0) rounds to, exact, as
// (m - 2^52) 2^-52 by integer operations (an FP64 instruction of a warp takes 64 cycles).
__device__ __forceinline__ double sym53(uint32_t hi, uint32_t lo) {
    const long long n = (long long)(((unsigned long long)hi << 21) | (unsigned long long)(lo >> 11)) - (1LL << 52);
    const unsigned long long a = (unsigned long long)(n < 0 ? -n : n);
    if (a == 0) return 0.0;
    const int z = __clzll((long long)a);  // a = 2^(63 - z) (1 + f): at most 53 bits, nothing is rounded
    const unsigned long long bits = ((unsigned long long)(1023 + 63 - z - 52) << 52) + (((a << z) >> 11) & 0x000FFFFFFFFFFFFFull);
    return __longlong_as_double((long long)(bits | (n < 0 ? 0x8000000000000000ull : 0ull)));
}

// Metropolis decision (Eq. 4) for dE with these bits and u = m 2^-53: accept iff dE <= 0 or u <
// exp(-beta dE). In FP32 first: p = __expf(-beta dE) is off by at most (2 + 1.2 |x|) 2^-23 p from the
// exponential of its argument (the intrinsic's documented bound), whose three roundings move it by
// |x| 3 2^-24 p, and u's 24 leading bits are below u by at most 2^-24; where the two sides are
// further apart than twice that the decision is the FP64 one, elsewhere it is taken in FP64.
__device__ __forceinline__ bool accept64(long long bits, double dE, double beta, float betaf, unsigned long long m) {
    if (bits <= 0) return true;  // dE <= 0 (or a negative NaN: the caller rejects NaN)
    const float x = -betaf * (float)dE, p = __expf(x), u = (float)(uint32_t)(m >> 29) * 0x1p-24f;
    const float tol = fmaf(p, (6.0f - 6.0f * x) * 0x1p-23f, 0x1p-22f);
    if (u > p + tol) return false;
    if (u < p - tol) return true;
    return __dmul_rn(__ull2double_rn(m), 0x1p-53) < exp(-dm(beta, dE));
}

// Point on the unit sphere by Marsaglia's method (Ann. Math. Stat. 43, 1972): draw
// (u1, u2) uniform in the square [-1, 1)^2 until s = u1^2 + u2^2 < 1, then
// (2 u1 sqrt(1-s), 2 u2 sqrt(1-s), 1 - 2 s). Candidate k uses counter word 3 = purpose|k.
__device__ double3 sphere64(uint32_t c0, uint32_t c1, uint32_t c2, uint32_t purpose, uint32_t k0, uint32_t k1,
                            uint32_t *err) {
    for (uint32_t k = 0; k < 64; ++k) {
        const uint4 w = philox10(make_uint4(c0, c1, c2, purpose | k), k0, k1);
        const double u1 = sym53(w.x, w.y), u2 = sym53(w.z, w.w);
        const double s = da(dm(u1, u1), dm(u2, u2));
        if (s >= 1.0) continue;
        const double q = __dsqrt_rn(ds(1.0, s));
        return make_double3(dm(dm(2.0, u1), q), dm(dm(2.0, u2), q), ds(1.0, dm(2.0, s)));
    }
    atomicOr(err, kErrSphere);
    return make_double3(0.0, 0.0, 1.0);
}

}  // namespace
}  // namespace vegas
