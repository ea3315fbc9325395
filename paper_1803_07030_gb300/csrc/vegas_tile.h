// The tiled cooperative sweep (vegas_tile.cu): its plan, arguments and launcher.
#pragma once

#include <cstdint>
#include <functional>
#include <memory>
#include <vector>

#include "vegas_internal.h"

namespace vegas {

constexpr int kTileThreads = 512;     // most sweeping threads per block
constexpr int kTileRecord = 128;      // threads of a block that form the MCS's totals
constexpr int kTilePerClass = 64;     // at least so many sites of the widest class per part: finer parts
                                      // only add boundary (29k-site core/shell particle, us per MCS: 4.9
                                      // with 32 to 64, 5.2 with 96 or 128, 6.3 with 256)
constexpr int kTileMcs = 1024;        // MCS per launch (bounds the buffer of the parts' totals)
constexpr int kTileCodes = 32;        // most exchange values of rows kept as words
constexpr int kTileRun = 64;          // most attempts of a thread per MCS (one FP32 run of its sums)

struct TilePart {
    int32_t own_begin, n_own;    // own sites: rows [own_begin, own_begin + n_own)
    int32_t halo_begin, n_halo;  // remote sites it reads: words halo_slot[halo_begin ..)
    int32_t site_begin;          // global sites of both, own first: site[site_begin ..)
    int32_t word_begin, n_words; // mailbox words of its own sites
};

struct TileClass {               // one colour class of one part, local site numbers
    int32_t begin, end;
    int32_t halo_begin, halo_end;
    int32_t lower_mode;          // 0: no link to a lower colour, 1: every link, 2: flagged per link
};

struct TileArgs {
    PassArgs pass;
    const TilePart *parts;       // [P]
    const TileClass *classes;    // [P][n_colours]
    const int32_t *site;         // global site of every local site of every part
    const int32_t *orig;         // caller id of every own site
    const int32_t *pub;          // mailbox word of every own site, -1 without a remote reader
    const int32_t *halo_slot;    // mailbox word of every remote site of every part
    const void *rows;            // [own site][width]: (local site | lower flag << 16, J) pairs, or words
    const float *codes;          // [n_codes] exchange values of a sample whose rows are words
    float4 *mail;                // [R][n_mail] (x, y, z, MCS counter + 1)
    double *partial;             // [mcs][R][4][P]
    uint32_t *count;             // [mcs][R][P] accepted attempts
    uint32_t *abort;             // set when a wait ran out: every block leaves, as do the run's later launches
    int64_t timeout_ns;
    uint32_t rk0[10], rk1[10];   // Philox round keys
    int32_t P, n_colours, n_mail, mcs, width;
    int32_t cubic;               // some site has a cubic constant
    int32_t skip_block;          // fault injection: this block never runs (-1: none)
    int32_t mem, n_codes, two_buffers;  // what is kept in shared memory (tile_shape)
    int32_t cap, rows_off, orig_off, pub_off, slot_off, code_off, cls_off, part_off;  // and where
};

struct TileShape {               // a loaded sample (new numbering) and the parts to cut it into
    int32_t n, n_colours, parts, width, site_off;
    const int32_t *cstart, *lower_mode, *col, *orig;
    const int64_t *row_ptr;
    const double *J;
};

struct TilePlan {
    std::vector<TilePart> parts;
    std::vector<TileClass> classes;
    std::vector<int32_t> site, orig, pub, halo_slot;
    std::vector<int32_t> part, local, word; // of every site (word: from its part's first, -1: none)
    std::vector<std::vector<int32_t>> own, halo;  // sites of every part
    std::unique_ptr<unsigned char[]> rows;  // pairs or words (tile_shape)
    size_t row_bytes = 0;
    std::vector<float> codes;               // exchange values
    int32_t n_mail = 0, max_own = 0, max_halo = 0, max_loc = 0, widest = 0;
    int32_t run = 0;                        // most attempts of one thread per MCS (tile_shape)
    bool columns = false;                   // a thread takes one site of each class, the same place in all
};

// Adds the exchange values J[0..n), as far as kTileCodes goes, and padding's 0.
void exchange_values(const double *J, int64_t n, std::vector<float> &values);
// The place of J in values (it is there); near: the last answer. Few values are compared without
// a branch, which the random signs of a spin glass would mispredict (0.3 ms for 20^3 sites).
inline uint32_t exchange_code(const std::vector<float> &values, float J, uint32_t near) {
    if (values.size() <= 4) {
        uint32_t c = 0;
        for (uint32_t k = 1; k < values.size(); ++k) c |= values[k] == J ? k : 0u;
        return c;
    }
    if (values[near] != J)
        for (near = 0; values[near] != J; ++near) {}
    return near;
}
// f(begin, end) for the chunks of [0, n), on several host threads.
void host_ranges(int64_t n, int32_t chunks, const std::function<void(int64_t, int64_t)> &f);
// False when the sample cannot be cut so.
bool tile_plan(const TileShape &s, TilePlan &out);
// Chooses the threads per block and what it keeps in shared memory, and writes the rows; 0 when
// the parts do not fit.
int tile_shape(TileArgs &a, const TileShape &s, TilePlan &p, size_t *smem);
void tile_tables(const TileArgs &a, const TileShape &s, TilePlan &p);  // the host side of those tables
int launch_tile_record(const TileArgs &a, void *stream);  // the records of a launch's MCS

// ---- FP64 (vegas_tile64.cu)
constexpr int kTile64Threads = 256;   // most sweeping threads per block
constexpr int kTile64Trial = 64;      // threads that draw trials
constexpr int kTile64Ahead = 4;       // classes of trials drawn ahead
constexpr int kTile64PerClass = 10;   // sites of the widest class per part
constexpr int kTile64Sites = 96;      // most sites of a class in a part

struct Tile64Trial {
    double x, y, z;        // trial spin
    unsigned long long u;  // acceptance uniform, u 2^-53
};

struct Tile64Args {
    TileArgs t;            // rows: words (local site | lower flag << 16); mail: two words per site
    const double *J;       // [own site][width]
    int32_t J_off, trial_off, widest;
};

// Threads that sweep, and the tables (J beside the plan's rows); 0 when the parts do not fit.
int tile64_shape(Tile64Args &a, const TileShape &s, TilePlan &p, std::vector<double> &J, size_t *smem);
int launch_tile64(const Tile64Args &a, int threads, size_t smem, void *stream);

// ---- batches with spins in shared memory (vegas_batch.cu)
constexpr int kBatchThreads = 512;    // sweeping threads per block
constexpr int kBatchColours = 30;     // most colour classes: a thread's FP32 sums of one MCS are then at most 64
                                      // attempts (spins in shared memory leave at most 34 sites per thread,
                                      // and one more per class), one run of the former kernels

struct BatchArgs {
    ResidentArgs r;
    const void *rows;            // [global site][kEllRow]: (site of the sample | lower flag << 16, J)
                                 // pairs, or words with J's index in codes from bit 17 on
    const float *codes;          // [n_codes]
    const int32_t *modes;        // [segment] 0: no link to a lower colour, 1: every link, 2: flagged
    uint32_t rk0[10], rk1[10];   // Philox round keys
    int32_t n_codes, cubic, clusters, part_off;
};

int batch_capacity(BatchArgs a, int cs, int sm_count);
int launch_batch(BatchArgs a, int n, int cs, void *stream);  // n clusters of cs blocks; the CUDA error

// Sweep of a.mcs MCS and their records; returns the CUDA error.
int launch_tile(const TileArgs &a, int threads, size_t smem, void *stream);

}  // namespace vegas
