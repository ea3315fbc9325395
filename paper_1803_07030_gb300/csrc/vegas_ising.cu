// Ising model with the spin-flip policy (Sec. II) on periodic square and simple cubic
// lattices, multi-spin coded: one 32-bit word holds 32 consecutive sites of one colour of
// one row (x direction) of one replica. A thread takes one word position (or, on small
// lattices, a part of it) for a group of four replicas, the four words of one Philox block per
// site: it compares every word with the acceptance thresholds of the step, which fills one
// bit mask per threshold, builds the count of neighbours aligned with each spin bit-sliced,
// and combines both into the flips of the 32 sites. Magnetization and bond sums are popcounts.
//
// Threshold: accept iff dE <= 0 or w < ceil(exp(-beta dE) 2^32), which for an integer w is
// exactly w 2^-32 < exp(-beta dE). The host computes exp in FP64 with the same expression
// as the definition, so the chain is the definition's bit for bit.
#include <cuda_runtime.h>

#include <algorithm>
#include <cmath>
#include <cstdint>
#include <cstring>
#include <new>
#include <string>
#include <vector>

#include "vegas_device.cuh"
#include "vegas_internal.h"

namespace vegas {
namespace {

constexpr uint32_t kPurposeIsing = 0x80000u;
constexpr uint32_t kPurposeIsingInit = 0x90000u;
constexpr int kIsingThreads = 256;
constexpr int kMaxIsingReplicas = 512;

// One threshold of one replica at one temperature/field step, with the spins it decides: those
// whose count of aligned neighbours has the bits selected by (x0, x1, x2) and whose own bit is
// selected by x3 (any when `any` is all ones). A class (own spin, aligned neighbours) whose flip is
// always accepted has no entry. Every field but neg is 0 or all ones.
struct __align__(16) IsingThr {
    uint32_t neg;         // 2^32 - thr: w + neg carries iff w >= thr (the flip is rejected)
    uint32_t x0, x1, x2;  // match = (p0 ^ x0) & (p1 ^ x1) & (p2 ^ x2) & (((own ^ x3) & on) | any)
    uint32_t x3, on, any;
    uint32_t never;       // thr = 0: rejected whatever w
};

struct IsingPassArgs {
    uint32_t *spins;
    const IsingThr *thr;      // [R][NQ] of this step
    unsigned long long *acc;  // [R][2]: up spins, aligned bonds (colour-1 ends) of the current MCS
    uint32_t *ticket;         // blocks done in the colour-1 pass (zero between passes)
    const double *h;          // [R] fields of this step
    double *hist;             // [R][2] record of this MCS
    double J;
    int64_t n;                // sites
    uint32_t rk0[10], rk1[10];  // Philox round keys (seed + r * Weyl constants)
    uint32_t t, rows, L, KW;  // MCS counter; rows = L^(dims-1), KW = L / 64 words per row and colour
    int32_t R, c, inst_base;
};

__host__ __device__ inline int64_t word_index(int r, int c, int64_t row, int kw, int64_t rows, int KW) {
    return ((int64_t)(r * 2 + c) * rows + row) * KW + kw;
}

// Adds the bit vector x to the bit-sliced counter (p0, p1, p2) (counts up to 7).
__device__ __forceinline__ void slice_add(uint32_t x, uint32_t &p0, uint32_t &p1, uint32_t &p2) {
    const uint32_t c0 = p0 & x;
    p0 ^= x;
    const uint32_t c1 = p1 & c0;
    p1 ^= c0;
    p2 ^= c1;
}

// R = 2R + carry(w + neg): appends the decision bit "w >= thr" to a mask in two instructions.
__device__ __forceinline__ void append_reject(uint32_t &mask, uint32_t w, uint32_t neg) {
    asm("{\n\t.reg .u32 s;\n\tadd.cc.u32 s, %1, %2;\n\taddc.u32 %0, %0, %0;\n\t}" : "+r"(mask) : "r"(w), "r"(neg));
}

// One colour pass. Bound by integer issue (Philox: 18 wide multiplies and 20 logic operations
// per site for four replicas; the spins are a bit each, so memory moves little). Every bit of the
// decision is therefore kept bit-sliced: two instructions per attempt and threshold (NQ = Z/2
// thresholds without a field, at most Z + 1 with one) in place of extracting the site's class
// and looking its threshold up. The random part needs no spin: it runs before
// griddepcontrol.wait, so it overlaps the tail of the pass before (programmatic dependent
// launch). S threads share a word position (32 / S sites each) on lattices too small to fill the
// GPU. 960^2 x 32 replicas: 90 us per MCS with class look-ups and a reduction kernel of its own
// (42 instructions per attempt), 27 us (1.08 T attempts/s) now.
template <int DIMS, int NQ, int S>
__global__ void __launch_bounds__(kIsingThreads) ising_pass_kernel(const IsingPassArgs a) {
    constexpr int Z = 2 * DIMS, NB = 32 / S;
    __shared__ uint32_t s_sum[8];
    __shared__ bool s_last;
    asm volatile("griddepcontrol.launch_dependents;" ::: "memory");
    if (threadIdx.x < 8) s_sum[threadIdx.x] = 0u;
    const uint32_t g = blockIdx.y, L = a.L, KW = a.KW, rows = a.rows, plane = rows * KW;
    const uint32_t idx = blockIdx.x * kIsingThreads + threadIdx.x;  // below 2^25 * 8 + 256
    const uint32_t item = idx / S, sub = idx % S;
    const bool active = item < plane;  // whole warps (plane is a multiple of 64)
    const int c = a.c, oc = 1 - c;
    uint32_t up[4] = {0u, 0u, 0u, 0u}, al[4] = {0u, 0u, 0u, 0u};
    __syncthreads();
    if (active) {
        const uint32_t row = item / KW, kw = item - row * KW;
        const uint32_t zc = DIMS == 3 ? row / L : 0u, y = row - zc * L;
        const uint32_t off = (y + zc + (uint32_t)c) & 1u;
        const IsingThr *T = a.thr + (size_t)g * 4 * NQ;
        uint32_t rej[4][NQ], neg[4][NQ];
#pragma unroll
        for (int j = 0; j < 4; ++j)
#pragma unroll
            for (int q = 0; q < NQ; ++q) {
                rej[j][q] = 0u;
                neg[j][q] = __ldg(&T[j * NQ + q].neg);
            }
        const uint32_t group = (uint32_t)(a.inst_base >> 2) + g;
        const uint32_t site0 = L * row + off + kw * 64u + 2u * NB * sub;  // x = 2 (32 kw + b) + off
#pragma unroll 2
        for (int b = NB - 1; b >= 0; --b) {  // the last appended bit is bit 0
            uint4 w = make_uint4(site0 + 2u * (uint32_t)b, a.t, group, kPurposeIsing);
#pragma unroll
            for (int r = 0; r < 10; ++r) {
                const uint32_t lo0 = 0xD2511F53u * w.x, hi0 = __umulhi(0xD2511F53u, w.x);
                const uint32_t lo1 = 0xCD9E8D57u * w.z, hi1 = __umulhi(0xCD9E8D57u, w.z);
                w = make_uint4(hi1 ^ w.y ^ a.rk0[r], lo1, hi0 ^ w.w ^ a.rk1[r], lo0);
            }
#pragma unroll
            for (int q = 0; q < NQ; ++q) {
                append_reject(rej[0][q], w.x, neg[0][q]);
                append_reject(rej[1][q], w.y, neg[1][q]);
                append_reject(rej[2][q], w.z, neg[2][q]);
                append_reject(rej[3][q], w.w, neg[3][q]);
            }
        }
        // every spin of the pass before is final from here on; read through L2, since a block of
        // that pass may have left older words in this SM's L1
        asm volatile("griddepcontrol.wait;" ::: "memory");
        const uint32_t rym = y == 0u ? row + L - 1u : row - 1u, ryp = y + 1u == L ? row + 1u - L : row + 1u;
        const uint32_t rzm = zc == 0u ? row + L * (L - 1u) : row - L, rzp = zc + 1u == L ? row - L * (L - 1u) : row + L;
        const uint32_t kws = off == 0u ? (kw == 0u ? KW - 1u : kw - 1u) : (kw + 1u == KW ? 0u : kw + 1u);
#pragma unroll
        for (int j = 0; j < 4; ++j) {
            uint32_t *So = a.spins + word_index((int)(g * 4) + j, c, 0, 0, rows, (int)KW);
            const uint32_t *Sn = a.spins + word_index((int)(g * 4) + j, oc, 0, 0, rows, (int)KW);
            const uint32_t own = __ldcg(So + item);
            const uint32_t xa = __ldcg(Sn + item), xb = __ldcg(Sn + row * KW + kws);
            uint32_t nb[Z];
            nb[0] = xa;                                                        // x neighbour at the same k
            nb[1] = off == 0u ? (xa << 1) | (xb >> 31) : (xa >> 1) | (xb << 31);  // k - 1 or k + 1
            nb[2] = __ldcg(Sn + rym * KW + kw);
            nb[3] = __ldcg(Sn + ryp * KW + kw);
            if (DIMS == 3) {
                nb[Z - 2] = __ldcg(Sn + rzm * KW + kw);
                nb[Z - 1] = __ldcg(Sn + rzp * KW + kw);
            }
            uint32_t p0 = 0u, p1 = 0u, p2 = 0u;
#pragma unroll
            for (int q = 0; q < Z; ++q) slice_add(~(own ^ nb[q]), p0, p1, p2);
            uint32_t reject = 0u;
#pragma unroll
            for (int q = 0; q < NQ; ++q) {
                const uint4 ta = __ldg((const uint4 *)&T[j * NQ + q]), tb = __ldg((const uint4 *)&T[j * NQ + q] + 1);
                const uint32_t match =
                    (p0 ^ ta.y) & (p1 ^ ta.z) & (p2 ^ ta.w) & (((own ^ tb.x) & tb.y) | tb.z);
                reject |= match & ((S > 1 ? rej[j][q] << (NB * sub) : rej[j][q]) | tb.w);
            }
#pragma unroll
            for (int o = 1; o < S; o <<= 1) reject |= __shfl_xor_sync(0xFFFFFFFFu, reject, o);
            const uint32_t flip = ~reject, nw = own ^ flip;
            if (S == 1 || sub == 0u) {
                if (flip) So[item] = nw;
                up[j] = (uint32_t)__popc(nw);
                // bonds aligned after the update, counted at their colour-1 ends: a aligned
                // neighbours stay a, or become Z - a under a flip
                if (c == 1)
                    al[j] = (uint32_t)(__popc(p0) + 2 * __popc(p1) + 4 * __popc(p2) + Z * __popc(flip) -
                                       2 * (__popc(p0 & flip) + 2 * __popc(p1 & flip) + 4 * __popc(p2 & flip)));
            }
        }
#pragma unroll
        for (int j = 0; j < 4; ++j) {
            const uint32_t u = __reduce_add_sync(0xFFFFFFFFu, up[j]);
            if ((threadIdx.x & 31) == 0) atomicAdd(&s_sum[2 * j], u);
            if (c == 1) {
                const uint32_t v = __reduce_add_sync(0xFFFFFFFFu, al[j]);
                if ((threadIdx.x & 31) == 0) atomicAdd(&s_sum[2 * j + 1], v);
            }
        }
    } else {
        asm volatile("griddepcontrol.wait;" ::: "memory");  // the counters below are the pass before's too
    }
    __syncthreads();
    if (threadIdx.x < 8 && s_sum[threadIdx.x])
        atomicAdd(&a.acc[(size_t)(g * 4 + threadIdx.x / 2) * 2 + (threadIdx.x & 1)], (unsigned long long)s_sum[threadIdx.x]);
    if (c == 0) return;
    // the colour-1 pass ends the MCS: its last block writes every replica's record (E, M) and
    // clears the counters (no other block touches them before this grid has ended)
    __threadfence();
    __syncthreads();
    if (threadIdx.x == 0) s_last = atomicAdd(a.ticket, 1u) == gridDim.x * gridDim.y - 1u;
    __syncthreads();
    if (!s_last) return;
    __threadfence();
    if (threadIdx.x == 0) *a.ticket = 0u;
    for (int r = (int)threadIdx.x; r < a.R; r += kIsingThreads) {
        const unsigned long long upc = __ldcg(&a.acc[r * 2]), alc = __ldcg(&a.acc[r * 2 + 1]);
        const int64_t M = 2 * (int64_t)upc - a.n;
        const int64_t bsum = 2 * (int64_t)alc - (int64_t)Z * (a.n / 2);
        a.hist[r * 2] = __dsub_rn(__dmul_rn(-a.J, (double)bsum), __dmul_rn(a.h[r], (double)M));
        a.hist[r * 2 + 1] = (double)M;
        a.acc[r * 2] = 0ull;
        a.acc[r * 2 + 1] = 0ull;
    }
}

// Initial state: bit 31 of the replica's word of Philox(seed; site, 0xFFFFFFFF, group, 0x90000).
__global__ void ising_init_kernel(uint32_t *S, uint64_t seed, int64_t rows, int32_t L, int32_t KW, int32_t R,
                                  int32_t dims, int32_t inst_base, int32_t all_up) {
    const int64_t per_g = rows * KW, n_items = 2 * (int64_t)(R / 4) * per_g;
    const uint32_t k0 = (uint32_t)seed, k1 = (uint32_t)(seed >> 32);
    for (int64_t item = (int64_t)blockIdx.x * blockDim.x + threadIdx.x; item < n_items;
         item += (int64_t)gridDim.x * blockDim.x) {
        const int c = (int)(item / ((int64_t)(R / 4) * per_g));
        const int64_t rest = item - (int64_t)c * (R / 4) * per_g;
        const int g = (int)(rest / per_g);
        const int64_t rem = rest - (int64_t)g * per_g;
        const int64_t row = rem / KW;
        const int kw = (int)(rem - row * KW);
        const int y = (int)(row % L), zc = dims == 3 ? (int)(row / L) : 0;
        const int off = (y + zc + c) & 1;
        uint32_t wd[4] = {0u, 0u, 0u, 0u};
        for (int b = 0; b < 32; ++b) {
            const uint32_t site = (uint32_t)((int64_t)L * row + off + (int64_t)kw * 64 + 2 * b);
            const uint4 w = philox10(make_uint4(site, 0xFFFFFFFFu, (uint32_t)(inst_base >> 2) + (uint32_t)g,
                                                kPurposeIsingInit),
                                     k0, k1);
            const uint32_t wj[4] = {w.x, w.y, w.z, w.w};
            for (int j = 0; j < 4; ++j) wd[j] |= (all_up ? 1u : (wj[j] >> 31)) << b;
        }
        for (int j = 0; j < 4; ++j) S[word_index(g * 4 + j, c, row, kw, rows, KW)] = wd[j];
    }
}

std::string g_ising_create_error;

}  // namespace
}  // namespace vegas

using namespace vegas;

struct vegas_ising {
    vegas_ising_options opt{};
    int device = 0, sm_count = 0;
    cudaStream_t stream = nullptr;
    bool own_stream = false;
    int64_t n = 0, rows = 0;
    int32_t KW = 0, Z = 0;
    uint32_t *d_spins = nullptr;
    IsingThr *d_thr = nullptr;
    uint32_t *d_ticket = nullptr;
    double *d_h = nullptr, *d_hist = nullptr;
    unsigned long long *d_acc = nullptr;
    size_t thr_cap = 0, hist_cap = 0;
    int split = 1;  // threads per word position
    std::vector<std::vector<double>> hist;  // per replica: records * 2
    int64_t records = 0;
    uint32_t t = 0;
    int64_t kernel_launches = 0, sweep_launches = 0, device_bytes = 0;
    double sweep_ms = 0.0, last_run_ms = 0.0;
    bool poisoned = false;
    std::string err;
};

namespace vegas {
namespace {

vegas_status ifail(vegas_ising *c, vegas_status st, const std::string &m) {
    if (c) {
        c->err = m;
        if (st == VEGAS_ECUDA || st == VEGAS_EDEVICE) c->poisoned = true;
    } else {
        g_ising_create_error = m;
    }
    return st;
}

// A host exception caught at an entry point, as a status (called inside a catch block).
vegas_status ising_host_exception(vegas_ising *c) {
    std::string m;
    const vegas_status st = status_of_current_exception(m);
    return ifail(c, st, m);
}

#define ICK(ctx, call)                                                                                 \
    do {                                                                                               \
        cudaError_t e_ = (call);                                                                       \
        if (e_ != cudaSuccess)                                                                         \
            return ifail((ctx), e_ == cudaErrorMemoryAllocation ? VEGAS_ENOMEM : VEGAS_ECUDA,          \
                         std::string(#call) + ": " + cudaGetErrorString(e_));                          \
    } while (0)

void ising_free(vegas_ising *c) {
    void *bufs[] = {c->d_spins, c->d_thr, c->d_ticket, c->d_h, c->d_hist, c->d_acc};
    for (void *b : bufs)
        if (b) cudaFree(b);
    if (c->own_stream && c->stream) cudaStreamDestroy(c->stream);
}

vegas_status ising_usable(vegas_ising *c) {
    if (!c) return VEGAS_EINVAL;
    if (c->poisoned) return VEGAS_ESTATE;
    return VEGAS_OK;
}

using IsingFn = void (*)(IsingPassArgs);

template <int DIMS, int NQ>
IsingFn select_split(int split) {
    if (split == 1) return ising_pass_kernel<DIMS, NQ, 1>;
    return split == 2 ? ising_pass_kernel<DIMS, NQ, 2> : split == 4 ? ising_pass_kernel<DIMS, NQ, 4> : ising_pass_kernel<DIMS, NQ, 8>;
}

// nq: thresholds per replica, Z / 2 or Z + 1.
cudaError_t launch_ising_pass(const vegas_ising *c, IsingPassArgs &a, int nq, int colour) {
    a.c = colour;
    const IsingFn f = c->opt.dims == 3 ? (nq == 3 ? select_split<3, 3>(c->split) : select_split<3, 7>(c->split))
                                       : (nq == 2 ? select_split<2, 2>(c->split) : select_split<2, 5>(c->split));
    cudaLaunchConfig_t cfg = {};
    cfg.gridDim = dim3((unsigned)((c->rows * c->KW * c->split + kIsingThreads - 1) / kIsingThreads), (unsigned)(a.R / 4));
    cfg.blockDim = dim3(kIsingThreads);
    cfg.stream = c->stream;
    cudaLaunchAttribute attr[1];
    attr[0].id = cudaLaunchAttributeProgrammaticStreamSerialization;
    attr[0].val.programmaticStreamSerializationAllowed = 1;
    cfg.attrs = attr;
    cfg.numAttrs = 1;
    return cudaLaunchKernelEx(&cfg, f, a);
}

// The thresholds of one replica at one step, into t[Z + 1]; returns how many there are. At most
// Z + 1: of the four classes with a or Z - a aligned neighbours (a < Z / 2), dE > 0 holds for at
// most two, and of the two with Z / 2 for at most one. Without a field the two spin directions
// share a threshold, which leaves Z / 2.
int ising_thresholds(double J, double beta, double hh, int Z, IsingThr *t) {
    uint32_t thr[2][8];
    bool always[2][8];
    for (int sb = 0; sb < 2; ++sb)
        for (int al = 0; al <= Z; ++al) {
            const double si = sb ? 1.0 : -1.0;
            const double sum = sb ? (double)(2 * al - Z) : (double)(Z - 2 * al);
            const double dE = 2.0 * si * (J * sum + hh);
            always[sb][al] = true;
            thr[sb][al] = 0u;
            if (dE <= 0.0) continue;
            // accept iff w < x = exp(-beta dE) 2^32 (w integer): iff w < ceil(x)
            const double x = std::ceil(std::exp(-(beta * dE)) * 4294967296.0);
            if (x >= 4294967296.0) continue;
            always[sb][al] = false;
            thr[sb][al] = (uint32_t)x;
        }
    int nq = 0;
    auto add = [&](int al, uint32_t x, uint32_t own1, uint32_t any) {
        IsingThr e{};
        e.neg = 0u - x;
        e.x0 = (al & 1) ? 0u : ~0u;
        e.x1 = (al & 2) ? 0u : ~0u;
        e.x2 = (al & 4) ? 0u : ~0u;
        e.x3 = own1 ? 0u : ~0u;
        e.on = ~0u;
        e.any = any;
        e.never = x == 0u ? ~0u : 0u;
        if (nq < Z + 1) t[nq] = e;
        ++nq;
    };
    for (int al = 0; al <= Z; ++al) {
        if (!always[0][al] && !always[1][al] && thr[0][al] == thr[1][al]) {
            add(al, thr[0][al], 0u, ~0u);
        } else {
            if (!always[0][al]) add(al, thr[0][al], 0u, 0u);
            if (!always[1][al]) add(al, thr[1][al], 1u, 0u);
        }
    }
    return nq;
}

}  // namespace
}  // namespace vegas

extern "C" void vegas_ising_default_options(vegas_ising_options *o) {
    if (!o) return;
    std::memset(o, 0, sizeof *o);
    o->dims = 2;
    o->L = 64;
    o->J = 1.0;
    o->replicas = 32;
    o->inst_base = 0;
    o->seed = 1;
    o->device = -1;
    o->cuda_stream = nullptr;
    o->init_up = 0;
    o->timing = 0;
}

// vegas_ising_create without the exception guard; *made is the context under construction.
static vegas_status ising_create(const vegas_ising_options *opt, vegas_ising **out, vegas_ising **made) {
    if (!out) return ifail(nullptr, VEGAS_EINVAL, "out is NULL");
    *out = nullptr;
    vegas_ising_options o;
    vegas_ising_default_options(&o);
    if (opt) o = *opt;
    if (o.dims != 2 && o.dims != 3) return ifail(nullptr, VEGAS_EINVAL, "dims must be 2 or 3");
    if (o.L < 64 || o.L % 64) return ifail(nullptr, VEGAS_EINVAL, "L must be a positive multiple of 64");
    const int64_t n = o.dims == 3 ? (int64_t)o.L * o.L * o.L : (int64_t)o.L * o.L;
    if (n >= ((int64_t)1 << 31)) return ifail(nullptr, VEGAS_EINVAL, "L^dims must be below 2^31");
    if (o.replicas < 4 || o.replicas > kMaxIsingReplicas || o.replicas % 4)
        return ifail(nullptr, VEGAS_EINVAL, "replicas must be a multiple of 4 in [4, 512]");
    if (o.inst_base < 0 || o.inst_base % 4) return ifail(nullptr, VEGAS_EINVAL, "inst_base must be a multiple of 4");
    if (!std::isfinite(o.J)) return ifail(nullptr, VEGAS_EINVAL, "J must be finite");
    if (o.init_up < 0 || o.init_up > 1 || o.timing < 0 || o.timing > 1)
        return ifail(nullptr, VEGAS_EINVAL, "init_up and timing must be 0 or 1");
    vegas_ising *c = new (std::nothrow) vegas_ising();
    if (!c) return ifail(nullptr, VEGAS_ENOMEM, "host allocation failed");
    *made = c;
    c->opt = o;
    c->n = n;
    c->rows = o.dims == 3 ? (int64_t)o.L * o.L : o.L;
    c->KW = o.L / 64;
    c->Z = 2 * o.dims;
    auto bail = [&](vegas_status st) {
        g_ising_create_error = c->err;
        ising_free(c);
        delete c;
        *made = nullptr;
        return st;
    };
    int ndev = 0;
    cudaError_t ce = cudaGetDeviceCount(&ndev);
    if (ce != cudaSuccess || ndev == 0) {
        c->err = std::string("no CUDA device: ") + cudaGetErrorString(ce);
        return bail(VEGAS_ECUDA);
    }
    if (o.device >= 0)
        c->device = o.device;
    else if (cudaGetDevice(&c->device) != cudaSuccess) {
        c->err = "cudaGetDevice failed";
        return bail(VEGAS_ECUDA);
    }
    vegas_status st;
    if ((st = [&]() -> vegas_status {
             ICK(c, cudaSetDevice(c->device));
             ICK(c, cudaDeviceGetAttribute(&c->sm_count, cudaDevAttrMultiProcessorCount, c->device));
             if (o.cuda_stream) {
                 c->stream = (cudaStream_t)o.cuda_stream;
             } else {
                 ICK(c, cudaStreamCreateWithFlags(&c->stream, cudaStreamNonBlocking));
                 c->own_stream = true;
             }
             const size_t words = (size_t)o.replicas * 2 * (size_t)c->rows * (size_t)c->KW;
             ICK(c, cudaMalloc(&c->d_spins, words * sizeof(uint32_t)));
             ICK(c, cudaMalloc(&c->d_ticket, sizeof(uint32_t)));
             ICK(c, cudaMalloc(&c->d_acc, sizeof(unsigned long long) * 2 * o.replicas));
             c->device_bytes = (int64_t)(words * 4 + sizeof(uint32_t) + 16 * (size_t)o.replicas);
             ICK(c, cudaMemsetAsync(c->d_acc, 0, sizeof(unsigned long long) * 2 * o.replicas, c->stream));
             ICK(c, cudaMemsetAsync(c->d_ticket, 0, sizeof(uint32_t), c->stream));
             const int64_t items = (int64_t)(o.replicas / 4) * c->rows * c->KW;
             // a thread per word position once they give every SM 16 warps; below, up to 8 threads
             // share one (a warp alone needs about 7 us for the 32 Philox blocks of a word)
             while (c->split < 8 && items * c->split < (int64_t)c->sm_count * 512) c->split *= 2;
             const int64_t init_items = 2 * items;
             const int ig = (int)std::min<int64_t>((init_items + 255) / 256, (int64_t)c->sm_count * 8);
             ising_init_kernel<<<ig, 256, 0, c->stream>>>(c->d_spins, o.seed, c->rows, o.L, c->KW, o.replicas, o.dims,
                                                          o.inst_base, o.init_up);
             ICK(c, cudaGetLastError());
             ICK(c, cudaStreamSynchronize(c->stream));
             c->kernel_launches = 1;
             return VEGAS_OK;
         }()) != VEGAS_OK)
        return bail(st);
    c->hist.assign((size_t)o.replicas, std::vector<double>());
    *out = c;
    return VEGAS_OK;
}

extern "C" vegas_status vegas_ising_create(const vegas_ising_options *opt, vegas_ising **out) {
    vegas_ising *made = nullptr;
    try {
        return ising_create(opt, out, &made);
    } catch (...) {
        const vegas_status st = ising_host_exception(nullptr);
        if (made) {
            ising_free(made);
            delete made;
        }
        if (out) *out = nullptr;
        return st;
    }
}

extern "C" vegas_status vegas_ising_run(vegas_ising *c, const double *T, const double *h, int32_t n_steps,
                                        int32_t mcs) {
    try {
        vegas_status st = ising_usable(c);
        if (st != VEGAS_OK) return st;
        if (n_steps < 0 || mcs < 0) return ifail(c, VEGAS_EINVAL, "n_steps and mcs_per_step must be >= 0");
        if (n_steps == 0 || mcs == 0) return VEGAS_OK;
        if (!T || !h) return ifail(c, VEGAS_EINVAL, "T or h is NULL");
        if ((int64_t)c->t + (int64_t)n_steps * mcs >= (int64_t)UINT32_MAX)
            return ifail(c, VEGAS_EINVAL, "global MCS counter would exceed 32 bits");
        const int R = c->opt.replicas, Z = c->Z;
        // thresholds [step][R][Z + 1], compacted below to each step's count
        std::vector<IsingThr> thr((size_t)n_steps * R * (Z + 1));
        std::vector<int> nq((size_t)n_steps, Z / 2);
        std::vector<double> hv((size_t)n_steps * R);
        for (int r = 0; r < R; ++r)
            for (int s = 0; s < n_steps; ++s) {
                const double Tv = T[(int64_t)r * n_steps + s], hh = h[(int64_t)r * n_steps + s];
                if (!(Tv > 0.0) || !std::isfinite(Tv)) return ifail(c, VEGAS_EINVAL, "T must be finite and > 0");
                if (!std::isfinite(hh)) return ifail(c, VEGAS_EINVAL, "h must be finite");
                const int k = ising_thresholds(c->opt.J, 1.0 / Tv, hh, Z, &thr[((size_t)s * R + r) * (Z + 1)]);
                if (k > Z + 1) return ifail(c, VEGAS_EINVAL, "more acceptance thresholds than classes with dE > 0");
                if (k > Z / 2) nq[(size_t)s] = Z + 1;
                hv[(size_t)s * R + r] = hh;
            }
        for (int s = 0; s < n_steps; ++s)
            if (nq[(size_t)s] == Z / 2)
                for (int r = 0; r < R; ++r)
                    for (int q = 0; q < Z / 2; ++q)
                        thr[(size_t)s * R * (Z + 1) + (size_t)r * (Z / 2) + q] = thr[((size_t)s * R + r) * (Z + 1) + q];
        ICK(c, cudaSetDevice(c->device));
        const int64_t nrec = (int64_t)n_steps * mcs;
        if (thr.size() > c->thr_cap) {
            if (c->d_thr) cudaFree(c->d_thr);
            if (c->d_h) cudaFree(c->d_h);
            c->d_thr = nullptr;
            c->d_h = nullptr;
            c->thr_cap = 0;
            ICK(c, cudaMalloc(&c->d_thr, sizeof(IsingThr) * thr.size()));
            ICK(c, cudaMalloc(&c->d_h, sizeof(double) * hv.size()));
            c->thr_cap = thr.size();
        }
        const size_t hneed = (size_t)nrec * R * 2;
        if (hneed > c->hist_cap) {
            if (c->d_hist) cudaFree(c->d_hist);
            c->d_hist = nullptr;
            c->hist_cap = 0;
            ICK(c, cudaMalloc(&c->d_hist, sizeof(double) * hneed));
            c->hist_cap = hneed;
        }
        ICK(c, cudaMemcpyAsync(c->d_thr, thr.data(), sizeof(IsingThr) * thr.size(), cudaMemcpyHostToDevice, c->stream));
        ICK(c, cudaMemcpyAsync(c->d_h, hv.data(), sizeof(double) * hv.size(), cudaMemcpyHostToDevice, c->stream));
        IsingPassArgs pa{};
        pa.spins = c->d_spins;
        pa.acc = c->d_acc;
        pa.ticket = c->d_ticket;
        pa.J = c->opt.J;
        pa.n = c->n;
        pa.rows = (uint32_t)c->rows;
        pa.L = (uint32_t)c->opt.L;
        pa.KW = (uint32_t)c->KW;
        pa.R = R;
        pa.inst_base = c->opt.inst_base;
        for (uint32_t q = 0; q < 10; ++q) {
            pa.rk0[q] = (uint32_t)c->opt.seed + q * 0x9E3779B9u;
            pa.rk1[q] = (uint32_t)(c->opt.seed >> 32) + q * 0xBB67AE85u;
        }
        std::vector<cudaEvent_t> ev;
        if (c->opt.timing) {
            ev.resize((size_t)nrec * 4);
            for (auto &x : ev) ICK(c, cudaEventCreate(&x));
        }
        cudaEvent_t e0, e1;
        ICK(c, cudaEventCreate(&e0));
        ICK(c, cudaEventCreate(&e1));
        ICK(c, cudaEventRecord(e0, c->stream));
        for (int64_t m = 0; m < nrec; ++m) {
            const int64_t s = m / mcs;
            pa.thr = c->d_thr + (size_t)s * R * (Z + 1);
            pa.h = c->d_h + s * R;
            pa.hist = c->d_hist + m * R * 2;
            pa.t = c->t + (uint32_t)m;
            for (int colour = 0; colour < 2; ++colour) {
                if (c->opt.timing) ICK(c, cudaEventRecord(ev[(size_t)m * 4 + 2 * colour], c->stream));
                ICK(c, launch_ising_pass(c, pa, nq[(size_t)s], colour));
                if (c->opt.timing) ICK(c, cudaEventRecord(ev[(size_t)m * 4 + 2 * colour + 1], c->stream));
            }
        }
        ICK(c, cudaGetLastError());
        ICK(c, cudaEventRecord(e1, c->stream));
        ICK(c, cudaStreamSynchronize(c->stream));
        float ms = 0.f;
        ICK(c, cudaEventElapsedTime(&ms, e0, e1));
        cudaEventDestroy(e0);
        cudaEventDestroy(e1);
        double sw = 0.0;
        for (size_t k = 0; k + 1 < ev.size(); k += 2) {
            float x = 0.f;
            ICK(c, cudaEventElapsedTime(&x, ev[k], ev[k + 1]));
            sw += x;
        }
        for (auto &x : ev) cudaEventDestroy(x);
        c->last_run_ms = ms;
        c->sweep_ms += sw;
        c->kernel_launches += nrec * 2;
        c->sweep_launches += nrec * 2;
        std::vector<double> hh(hneed);
        ICK(c, cudaMemcpy(hh.data(), c->d_hist, sizeof(double) * hneed, cudaMemcpyDeviceToHost));
        for (int r = 0; r < R; ++r) {
            auto &v = c->hist[(size_t)r];
            const size_t old = v.size();
            v.resize(old + (size_t)nrec * 2);
            for (int64_t k = 0; k < nrec; ++k) {
                v[old + (size_t)k * 2] = hh[((size_t)k * R + r) * 2];
                v[old + (size_t)k * 2 + 1] = hh[((size_t)k * R + r) * 2 + 1];
            }
        }
        c->records += nrec;
        c->t += (uint32_t)nrec;
        return VEGAS_OK;
    } catch (...) {
        return ising_host_exception(c);
    }
}

extern "C" vegas_status vegas_ising_history(const vegas_ising *cc, double *out, size_t capacity, size_t *n_written) {
    try {
        vegas_ising *c = const_cast<vegas_ising *>(cc);
        vegas_status st = ising_usable(c);
        if (st != VEGAS_OK) return st;
        const size_t need = (size_t)c->opt.replicas * (size_t)c->records * 2;
        if (n_written) *n_written = need;
        if (!out) return VEGAS_OK;
        if (capacity < need) return ifail(c, VEGAS_EINVAL, "history buffer too small");
        for (int r = 0; r < c->opt.replicas; ++r)
            std::memcpy(out + (size_t)r * c->records * 2, c->hist[(size_t)r].data(), sizeof(double) * c->records * 2);
        return VEGAS_OK;
    } catch (...) {
        return ising_host_exception(const_cast<vegas_ising *>(cc));
    }
}

namespace vegas {
namespace {

// Copies one replica's words (both colours) between device and host, then (un)packs them.
vegas_status ising_spins_io(vegas_ising *c, int32_t replica, int8_t *out, const int8_t *in) {
    vegas_status st = ising_usable(c);
    if (st != VEGAS_OK) return st;
    if (replica < 0 || replica >= c->opt.replicas) return ifail(c, VEGAS_EINVAL, "replica out of range");
    ICK(c, cudaSetDevice(c->device));
    const int L = c->opt.L, KW = c->KW;
    const int64_t rows = c->rows;
    std::vector<uint32_t> w((size_t)2 * rows * KW);
    uint32_t *dev = c->d_spins + word_index(replica, 0, 0, 0, rows, KW);
    if (in)
        for (int64_t i = 0; i < c->n; ++i)
            if (in[i] != 1 && in[i] != -1) return ifail(c, VEGAS_EINVAL, "spins must be +1 or -1");
    if (out) ICK(c, cudaMemcpy(w.data(), dev, sizeof(uint32_t) * w.size(), cudaMemcpyDeviceToHost));
    for (int col = 0; col < 2; ++col)
        for (int64_t row = 0; row < rows; ++row) {
            const int y = (int)(row % L), zc = c->opt.dims == 3 ? (int)(row / L) : 0;
            const int off = (y + zc + col) & 1;
            for (int kw = 0; kw < KW; ++kw) {
                uint32_t &word = w[(size_t)(((int64_t)col * rows + row) * KW + kw)];
                for (int b = 0; b < 32; ++b) {
                    const int64_t site = (int64_t)L * row + off + 64 * kw + 2 * b;
                    if (out)
                        out[site] = ((word >> b) & 1u) ? 1 : -1;
                    else if (in[site] > 0)
                        word |= 1u << b;
                }
            }
        }
    if (in) {
        ICK(c, cudaMemcpy(dev, w.data(), sizeof(uint32_t) * w.size(), cudaMemcpyHostToDevice));
    }
    return VEGAS_OK;
}

}  // namespace
}  // namespace vegas

extern "C" vegas_status vegas_ising_get_spins(const vegas_ising *c, int32_t replica, int8_t *out) {
    try {
        if (!out) return ifail(const_cast<vegas_ising *>(c), VEGAS_EINVAL, "out is NULL");
        return ising_spins_io(const_cast<vegas_ising *>(c), replica, out, nullptr);
    } catch (...) {
        return ising_host_exception(const_cast<vegas_ising *>(c));
    }
}

extern "C" vegas_status vegas_ising_set_spins(vegas_ising *c, int32_t replica, const int8_t *in) {
    try {
        if (!in) return ifail(c, VEGAS_EINVAL, "in is NULL");
        return ising_spins_io(c, replica, nullptr, in);
    } catch (...) {
        return ising_host_exception(c);
    }
}

extern "C" vegas_status vegas_ising_set_mcs_counter(vegas_ising *c, uint32_t t) {
    try {
        vegas_status st = ising_usable(c);
        if (st != VEGAS_OK) return st;
        if (t == UINT32_MAX) return ifail(c, VEGAS_EINVAL, "MCS counter must be below 2^32 - 1");
        c->t = t;
        return VEGAS_OK;
    } catch (...) {
        return ising_host_exception(c);
    }
}

extern "C" vegas_status vegas_ising_stats(const vegas_ising *c, vegas_stats_t *o) {
    try {
        if (!c || !o) return VEGAS_EINVAL;
        std::memset(o, 0, sizeof *o);
        o->n_samples = 1;
        o->n_instances = c->opt.replicas;
        o->replicas = c->opt.replicas;
        o->max_colours = 2;
        o->n_sites = c->n;
        o->n_edges = c->n * c->Z;
        o->records = c->records;
        o->mcs_done = c->t;
        o->kernel_launches = c->kernel_launches;
        o->sweep_launches = c->sweep_launches;
        o->sweep_ms = c->sweep_ms;
        o->last_run_ms = c->last_run_ms;
        o->device_bytes = c->device_bytes;
        return VEGAS_OK;
    } catch (...) {
        return ising_host_exception(const_cast<vegas_ising *>(c));
    }
}

extern "C" const char *vegas_ising_last_error(const vegas_ising *c) {
    if (!c) return g_ising_create_error.c_str();
    return c->err.c_str();
}

extern "C" void vegas_ising_destroy(vegas_ising *c) {
    if (!c) return;
    cudaSetDevice(c->device);
    if (c->stream) cudaStreamSynchronize(c->stream);
    ising_free(c);
    delete c;
}
