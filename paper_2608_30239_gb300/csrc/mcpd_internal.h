// Private declarations shared by the host table builder, the C ABI and the CUDA kernels.
#pragma once
#include <stdint.h>

#include <algorithm>
#include <string>
#include <vector>

#include <cuda_runtime_api.h>

#include "../../include/mcpd.h"

// A context: one device, one stream.  Defined here so every translation unit of the library
// sees the same definition.
struct mcpd_ctx {
    int device = 0;
    cudaStream_t stream = nullptr;
    int sm_count = 0;
    size_t smem_optin = 0;
    std::string err;
    // Staging of mcpd_features_batch, kept between calls up to kKeepStaging bytes: pinned host memory
    // and device memory of the same size.
    void *stage_host = nullptr, *stage_dev = nullptr;
    size_t stage_bytes = 0;
};

namespace mcpd {

constexpr size_t kKeepStaging = size_t(32) << 20;

constexpr int kRow = 8;              // pool entries per clone row (one 16-byte shared load)
constexpr int kTSide = kRow + 1;     // acceptance table is kTSide x kTSide, indexed 9 n+ + n-
constexpr int kMaskDeg = 6;          // uniform degrees up to this use mask-indexed thresholds
constexpr int kBank = 96;            // slots of a chunk, at most
constexpr int kMaxClones = 65535;
constexpr int kMaxPools = 1022;      // pool byte offsets must fit 16 bits
constexpr int kMaxPoolSize = 255;    // per-pool counts are bytes
constexpr int64_t kMaxBuckets = 1 << 16;

// Counter slots of the device statistics block.
enum Counter {
    kWork = 0, kProgress, kSiteUpdates, kRepsStarted, kRepsRetained, kRepsAborted,
    kZeroCompletion, kStepLimitHits, kMaxTau, kSumTau, kTauOverAudit, kNumCounters = 16
};

// Per-lane statistics record of the sampling kernel, summed into the counters at exit.
enum PairStat {
    kPsProgress = 0, kPsStarted, kPsRetained, kPsAborted, kPsZero, kPsLimit, kPsSumTau, kPsMaxTau,
    kPsTauAudit, kPsSiteUpdates, kPairStats = 10
};

// Lane-group kernel: per-pair scratch, one contiguous block of 8-byte words per pair: the
// replication's and the slot's sums G in two halves of [0, 2 na), kPairStats words it leaves unused,
// then the touched-clone bit sets of the replication and of the slot (W 32-bit words each).
#ifdef __CUDACC__
#define MCPD_HD __host__ __device__
#else
#define MCPD_HD
#endif
MCPD_HD inline long long pair_words(long long na, long long W) { return 2 * na + kPairStats + W; }
// Sampling kernel: an entry is one slot's sums G [na] and `marks` words for the bit set of the clones
// touched (mark_words); a warp's scratch is `bank` entries, the list of those whose pairs are done (two
// 32-bit words each), a statistics record per lane and, coupled, an entry per pair (at most 16, and one
// per slot of a chunk).  In 8-byte words.
MCPD_HD inline long long warp_words(long long bank, long long na, long long marks, bool coupled) {
    return (bank + (coupled ? (bank < 16 ? bank : 16) : 0)) * (na + marks) + bank + 32 * kPairStats;
}
#undef MCPD_HD
// Words of an entry's marks: W 32-bit words and one for `all` (some event was not marked), or none.  A
// slot of few steps touches few of its clones, and reading all na sums for it costs more than its steps
// do; in small instances, or with many flips, a mark per event costs more than the reading.  Uncoupled, all
// sums against marks: 5000 clones, 80,000 slots of 52 steps 2.4 -> 0.2 to 0.3 ms, of a sweep 5.6 -> 4; 1298
// clones, of 52 steps 0.6 -> 0.3 to 0.5, of two sweeps 2.8 -> 2.3; 600 clones from 0.53 -> 0.37 (6 steps) to 0.66 ->
// 0.92 (60 steps, low noise), equal at two sweeps; 333 clones mostly slower (0.89 -> 2.1 ms at worst).  Coupled:
// 5000 clones, 9 to 800 steps 7 to 9 -> 2.2 to 3.7 ms; 2500 clones 10 to 30% less; 1298 the same.  Longer slots of
// large instances would gain too (2500 clones, five sweeps 7.8 -> 6.7 ms).
// steps, clones: sums over the launch's slots; a pair marks its first half sweep (mark_steps keeps out lags
// beyond it).
inline double mark_steps(bool coupled, int64_t B, int64_t unit, int64_t lag) {
    return static_cast<double>(coupled ? std::max(std::max(B, unit), 2 * lag) : std::max(B, unit));
}
inline int32_t mark_words(bool coupled, double steps, double clones, int32_t max_na, int32_t W) {
    return steps < (coupled ? 1.0 : 2.0) * clones && max_na >= (coupled ? 2048 : 512) ? (W + 2) / 2 : 0;
}

// Threads per block the sampling kernel is compiled for: 20 warps of 96 registers, and 16 of 128 for the
// builds with eight row entries or a batch's descriptors.  More warps lose more to the registers they
// take than they hide: 24 warps of 80 registers against 20 of 96, 1298 x 97 at high noise, 105.5 against
// 94.7 ms (low noise 24.9 and 22.3, a learned start 21.0 and 18.3); 18 of 112: 103.4 ms; 16 of 128:
// 108.4.  Batches at 20 of 96 against 16 of 128: 128 uneven instances 67.0 against 60.8 ms.
constexpr int pairs_threads(int deg, bool batch) { return batch || deg == 0 || deg > kMaskDeg ? 512 : 640; }

// Everything the sampler needs, built on the host from (design, y, params).
struct Tables {
    int32_t n = 0, m = 0, na = 0, deg_max = 0;
    int32_t scan = MCPD_SCAN_SCORE;
    bool coupled = true;
    std::vector<int32_t> active;      // [na] original index of active clone a, ascending
    std::vector<uint64_t> alias;      // [na] prob (low 32) | alias index (high 32)
    std::vector<uint16_t> rows;       // [na * kRow] byte offsets of the pools' counts: see build_tables
    std::vector<uint16_t> rows_pool;  // [na * kRow] pool id | y << 15, 0xFFFF past the clone's pools
    std::vector<uint64_t> T;          // [kTSide * kTSide]
    std::vector<uint64_t> Tnu;        // [na] or empty
    std::vector<uint32_t> init_pairs; // even clone ids a with Tnu[a] or Tnu[a+1] nonzero
    std::vector<double> w;            // [na] scan weights
    std::vector<uint16_t> rows_mask;  // [na * kRow] uniform degree <= kMaskDeg: see build_tables
    std::vector<uint64_t> T_mask;     // [(kMaskDeg + 1) * 64] or empty
    // shared-memory layout of one pair (32-bit words, interleaved over the 32 lanes of a warp)
    int32_t udeg = 0;                 // d if every active clone sits in exactly d pools, else 0
    int32_t W = 0;                    // bit-set words per chain
    int32_t Mp = 0;                   // count words (four pools per word, the padding pool included)
    int32_t wpp = 0;                  // words per column = W + Mp (one chain)
    uint16_t dummy_entry = 0;         // row entry of the padding pool
    uint32_t dummy_word = 0;          // initial value of the word holding the padding pool
    int32_t dummy_word_index = 0;
    // run shape
    int64_t k = 0, ell = 0, L = 0, burn = 0, length = 0, unit = 1;
    int64_t P = 0, B = 0, nb = 1, step_limit = 0, slot_offset = 0, trace_stride = 0, tau_audit = 0;
    bool capped = false;              // meeting cap: step_limit is the cap, a capped pair is kept
    int64_t lag = 1;                  // coupled lag L
    int64_t trace_steps = 0, trace_reps = 0;   // per-replication trajectory records (tests)
    uint64_t seed = 0;
    uint32_t instance = 0;
    bool record_slots = false;
};

int build_tables(const mcpd_design *design, const uint8_t *y, const mcpd_params *params,
                 Tables *out, std::string *err);

// The run's counters (summed over launches) as mcpd_stats; n_buckets, n_active and kernel_ms are
// the caller's.
inline void counters_to_stats(const unsigned long long *c, mcpd_stats *s) {
    s->progress_units = static_cast<int64_t>(c[kProgress]);
    s->site_updates = static_cast<int64_t>(c[kSiteUpdates]);
    s->reps_started = static_cast<int64_t>(c[kRepsStarted]);
    s->reps_retained = static_cast<int64_t>(c[kRepsRetained]);
    s->reps_aborted = static_cast<int64_t>(c[kRepsAborted]);
    s->zero_completion_slots = static_cast<int64_t>(c[kZeroCompletion]);
    s->step_limit_hits = static_cast<int64_t>(c[kStepLimitHits]);
    s->max_tau = static_cast<int64_t>(c[kMaxTau]);
    s->sum_tau = static_cast<int64_t>(c[kSumTau]);
    s->tau_over_audit = static_cast<int64_t>(c[kTauOverAudit]);
}

// The rows and thresholds the single-instance kernel stages (mask-indexed when available).
inline const std::vector<uint16_t> &kernel_rows(const Tables &t) { return t.rows_mask.empty() ? t.rows : t.rows_mask; }
inline const std::vector<uint64_t> &kernel_T(const Tables &t) { return t.T_mask.empty() ? t.T : t.T_mask; }
inline size_t kernel_table_bytes(const Tables &t) {
    return (static_cast<size_t>(t.na) * 24 + kernel_T(t).size() * 8 + 15) / 16 * 16;
}

// Kernel arguments (plain types only: shared by host and device compilation units).
struct KParams {
    const uint64_t *alias;
    const uint16_t *rows;
    const uint64_t *T;
    const uint64_t *Tnu;
    const uint32_t *init_pairs;       // [n_init_pairs]
    int32_t n_init_pairs;
    long long *pair_scratch;          // [warps][warp_words(bank, na, marks, coupled)]
    unsigned long long *S1;           // [nb][na]
    unsigned long long *S2lo;         // [nb][na]
    unsigned long long *S2hi;         // [nb][na]
    unsigned long long *bcount;       // [nb]
    unsigned long long *counters;     // [kNumCounters]
    int *error;
    int32_t *slot_nstar;
    long long *slot_S;
    int32_t *slot_reps;
    long long *trace_G;
    int32_t na, m, W, Mp, wpp, deg, nb, scan;
    int32_t udeg, capped;             // uniform degree (0: mixed); 1: the step limit is a meeting cap
    uint32_t dummy_entry, dummy_word;
    int32_t dummy_word_index, coupled;
    long long P, B, k, ell, L, burn, length, unit, step_limit, slot_offset, trace_stride, tau_audit;
    unsigned long long seed;
    uint32_t instance;
    int32_t warps;
    uint32_t smem_tables;             // bytes of staged tables at the start of shared memory
    int32_t bank, chunk;              // entries per warp; slots a warp takes at a time (<= bank)
    int32_t marks;                    // words of marks per entry
    uint32_t rk[20];                  // Philox round keys of the seed
    int32_t nT;                       // threshold entries staged (kTSide^2, or mask-indexed)
    int32_t lag;                      // coupled lag L >= 1
    int32_t *trace_rec;               // [n_trace][trace_reps][4 + trace_steps] or null
    int32_t trace_reps, trace_steps;
};

// Philox4x32-10 round keys of a 64-bit seed: (lo + i 0x9E3779B9, hi + i 0xBB67AE85), i = 0..9.
inline void philox_round_keys(uint64_t seed, uint32_t rk[20]) {
    uint32_t k0 = static_cast<uint32_t>(seed), k1 = static_cast<uint32_t>(seed >> 32);
    for (int i = 0; i < 10; ++i) {
        rk[2 * i] = k0;
        rk[2 * i + 1] = k1;
        k0 += 0x9E3779B9u;
        k1 += 0xBB67AE85u;
    }
}

// One instance of a batched launch (plain types; read by the kernels from global memory).
struct InstDesc {
    const uint64_t *alias;            // [na]
    const uint16_t *rows;             // [na * kRow] count offsets for the interleaved pair layout
    const uint64_t *T;                // [kTSide * kTSide]
    const uint64_t *Tnu;              // [na] or null
    const uint32_t *init_pairs;       // [n_init_pairs] even clone ids with a nonzero threshold
    const uint16_t *rows_pool;        // [na * kRow] pool id | y << 15 (lane-group kernels)
    const uint16_t *rows_mask;        // [na * kRow] mask-indexed rows (uniform degree 3..kMaskDeg) or null
    const uint64_t *T_mask;           // [(kMaskDeg + 1) * 64] or null
    unsigned long long *S1, *S2lo, *S2hi, *bcount;   // this instance's N*_p buckets
    int32_t n_init_pairs, capped;     // capped: the step limit is a meeting cap
    int32_t na, W, wpp, deg, nb, dummy_word_index;
    uint32_t dummy_entry, dummy_word;
    long long P, B, k, ell, L, burn, length, unit, step_limit, slot_offset, tau_audit;
    long long work_begin;             // global index of this instance's first slot in the launch
    long long unit_begin, units;      // its chunks in the launch: the first one's index, their number
    long long P_total;                // slots in this instance's buckets (the finalize's P)
    unsigned long long seed;
    uint32_t instance;
    int32_t lag;                      // coupled lag L >= 1
};

// Arguments of a batched launch.
struct BParams {
    const InstDesc *insts;
    int32_t n_inst, coupled, scan, max_wpp;
    int32_t lanes, max_m;             // lanes per pair (1, 8, 16, 32); largest pool count
    long long total_work, total_units;   // slots; chunks
    long long *pair_scratch;          // [warps][warp_words(bank, max_na, marks, coupled)], or per pair pair_words (lane groups)
    unsigned long long *counters;
    int *error;
    int32_t max_na, max_W;
    int32_t bank;                     // entries per warp (the slots of a chunk, at most)
    int32_t marks;                    // words of marks per entry
    int32_t ext;                      // some instance has a meeting cap or a lag > 1
    int32_t udeg;                     // every instance of the class has this uniform degree (0: mixed)
};

// Launch shape of the sampling kernel (mcpd_kernels.cu).
struct PairsShape {
    int warps = 0;                    // warps per block
    int per_sm = 1;                   // resident blocks per SM
    size_t smem = 0;                  // dynamic shared memory per block
};
inline size_t pairs_smem_bytes(size_t tables, int wpp, int warps) {
    return (tables + static_cast<size_t>(warps) * static_cast<size_t>(wpp) * 128 + 15) / 16 * 16;
}
// How `slots` slots are run on `blocks` resident blocks of at most `most` warps: warps per block and
// slots a warp takes at a time (a chunk).  All of a warp's share at once (in equal parts if a bank
// cannot hold it): a chunk's single runs are dealt to the lanes one by one, so any number of slots fills
// them, and its pairs fill a warp the better the more there are.  All warps once the slots give each
// 16 pairs; below that at most kSpreadWarps per block, since the time of few slots is their pairs':
// 16384 slots with a lag of one sweep take 14.5, 14.5, 15.8 and 17.9 ms on at most 8, 12, 16 and 20 warps
// (4096 slots 10.2, 11.7, 13.2, 15.6; without the lag 16384 slots 5.7, 5.3, 5.3, 5.6; 1298 x 97, high noise).
constexpr int kSpreadWarps = 12;
struct ChunkShape { int warps, chunk; };
inline ChunkShape chunk_shape(long long slots, long long blocks, int most, long long bank) {
    auto up = [](long long a, long long b) { return (a + b - 1) / b; };
    const long long w = std::min<long long>(most, std::max(up(slots, blocks * 16), std::min<long long>(kSpreadWarps, up(slots, blocks))));
    const long long share = up(slots, blocks * w);
    return {static_cast<int>(w), static_cast<int>(up(share, up(share, bank)))};
}
// tables: bytes staged at the start of shared memory (0 for batches); wpp: words per column;
// P: slots of a single instance (0: as many warps as fit); warps: requested warps (0 = auto); marks:
// the builds with marks.
int pairs_shape(int coupled, int scan, int udeg, bool batch, size_t tables, int wpp, size_t smem_optin,
                long long P, int sm_count, int warps, bool ext, bool marks, PairsShape *out);

// The batched sampling-kernel variants (mcpd_batch.cu): the kernel for a class, and the
// compile-time degree a class of uniform degree udeg runs with (0: the generic build).
using PairsKernelFn = void (*)(const KParams, const BParams);
PairsKernelFn pick_batch(int coupled, int scan, int udeg);
PairsKernelFn pick_marks(int coupled, int scan, bool batch, int udeg);   // the builds with marks (mcpd_marks.cu)
PairsKernelFn pick_batch_marks(int coupled, int scan, int udeg);         // (mcpd_batch_marks.cu)
PairsKernelFn pick_batch_degree(int udeg);                  // coupled, degrees 4, 5, 7, 8 (mcpd_batch_deg.cu)
int batch_kernel_degree(int coupled, int ext, int udeg);

// Launchers (mcpd_kernels.cu).
int launch_batch(const BParams &bp, int grid, int block, size_t smem, void *stream);
int launch_group(const BParams &bp, int grid, int block, size_t smem, void *stream);
int set_group_smem(int lanes, size_t bytes);
int group_max_threads(int lanes);
int group_occupancy(int lanes, int block, size_t smem, int *blocks_per_sm);
int launch_finalize_batch(const InstDesc *insts, int n_inst, const int32_t *clone_inst,
                          const int32_t *clone_local, long long total_clones, double *est,
                          double *se, void *stream);
int launch_pairs(const KParams &kp, int grid, int block, size_t smem, void *stream);
// The recording variants (mcpd_trace.cu): launched by launch_pairs when kp.trace_rec is set.
int launch_pairs_trace(const KParams &kp, int grid, int block, size_t smem, void *stream);
int launch_finalize(const unsigned long long *S1, const unsigned long long *S2lo,
                    const unsigned long long *S2hi, int na, int nb, long long P, long long L,
                    double *est, double *se, void *stream);
int launch_philox(const uint32_t *ctr, uint32_t k0, uint32_t k1, uint32_t *out, long long n,
                  void *stream);
int pairs_max_smem(int device, size_t *bytes);

}  // namespace mcpd
