// The order in which the FP32 sweeps add their attempts, as far as the choice of a sweep depends on it.
//
// Every sweep adds the attempts' shares of (E, Mx, My, Mz) in FP32 along a thread, class after class,
// and the threads' sums in FP64. A thread of the resident, cooperative and cluster sweeps takes every
// at_once-th site of a class. Sweeps of one sample that give a thread the same sites agree to the
// FP64 sums' rounding; others differ by the FP32 sums' rounding, about 3e-8 k / sqrt(n) of the
// record at T = 2 for threads of k attempts and n sites (3e-9 with 1,690 sites on 512 threads, 1.3e-9
// with 10,648 sites x 16 replicas). A context chosen automatically records the sums of the sweep
// that the library's first kernels make fastest: a faster kernel takes that sweep's place only where
// it adds in its order.
#pragma once

#include <cstdint>

namespace vegas {

struct TileOrder {
    bool columns;      // a thread of the tiled sweep takes one site of each class, the same place in all
    int64_t widest;    // sites of the widest class
    int64_t n;         // sites
    int32_t replicas;
    int32_t run;       // most attempts of one thread of the tiled sweep per MCS
};

// Whether the tiled sweep may take the place of sweep v (1 resident, 2 cooperative, 3 cluster), which
// gives its threads at_once sites of a class at a time: in its order, or, with one replica in parts of several
// rounds (150,000 sites and more on a whole GPU), where the records agree to 4e-10 up to T = 2 and to
// 1e-9 at T = 6 (64^3 at T = 0.5, 128^3 at T = 0.8: 2.4e-10 and 2.9e-10) and the tiled sweep runs two to three times
// faster. Several replicas leave a part fewer sites to average over: 5e-10 with 2 or 4, 9e-10 with 8 and
// 1.3e-9 with 16 (T = 2), so there the other sweep stays.
inline bool tile_in_order(const TileOrder &t, int v, int64_t at_once) {
    if (v < 1 || v > 3) return false;
    if (t.columns && t.widest <= at_once) return true;
    return v == 2 && t.replicas == 1 && 1600 * (int64_t)t.run * t.run <= t.n;
}

// The time at which the autotuner compares the per-class sweep: that of its first kernels, whose
// records (one FP32 run per class, or with 32 replicas in no fixed order) then stand for the context's. us per
// MCS, then and now: 4 more for the reduction (25.1 and 21.1 at 25,200 sites, 48.3 and 42.7 at 30,482 x 16), and
// with the kernel of 32 replicas 1.12 t + 6 (56.0 and 45.4 at 22,736 sites, 64.6 and 56.2 at 39,200, 90 and 70 at
// 127,449, 106 and 89 at 148,877). On 60 glasses and ferromagnets of 13,000 to 330,000 sites x 32 the
// choice is the former one but for four whose times were within 5% of each other.
inline double per_class_us(double us, bool kernel_of_32) { return kernel_of_32 ? 1.12 * us + 6.0 : us + 4.0; }

}  // namespace vegas
