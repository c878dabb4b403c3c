// The persistent sampling kernel (template): a warp runs a chunk of slots, each slot's pairs to
// their meetings first and its single chains after (Algorithms 3 and 4).  Included by the
// translation units that instantiate it: mcpd_kernels.cu and mcpd_batch*.cu (the production
// variants), mcpd_marks.cu and mcpd_batch_marks.cu (MARKS: slots of few steps, see mark_words) and
// mcpd_trace.cu (TRACE: the variants that also record per-replication trajectories).
#pragma once
#include <cuda_runtime.h>
#include <stdint.h>

#include "mcpd_device.cuh"
#include "mcpd_internal.h"

namespace mcpd {
namespace {

// The estimator's integer bookkeeping.  Swapping the sums in
// L H_{k:l} = sum_{r=k}^{l} [X_r + sum_{s>=1} (X_{r+s} - Y_{r+s-1})] gives
//   G_j = sum_{t=0}^{C} w(t) X_t[j] - sum_{t=0}^{C-1} w(t) Y_t[j],  w(t) = clamp(t - k + 1, 0, L),
// so a chain whose bit j is 1 on the time interval [s, e] contributes +-(W(e) - W(s-1)) with
// W(u) = sum_{v<=u} w(v).  In events: X flips at step t add -+W(t), Y flips +-W(t-1), and the open
// intervals close at C.  Splitting W(t) = w(t) + W(t-1) splits G into
//   (a) a sum over X alone: every X flip adds -+w(t), and a bit of X_C adds w(C);
//   (b) a correction over t < tau: X flips add -+W(t-1) and Y flips +-W(t-1); from the meeting on
//       X_{t} = Y_{t-1} and the two cancel.
// w is constant (L) from t = l on, so in (a) a flip at t >= l and its closing term cancel: (a) is
// the same for every C >= l, and X need only be run for l steps, whatever tau.  With lag L_g the
// split is W(t) = w(t) + W(t-L_g), w the one-lag count of window indices r <= t, and a pair stopped
// unmet at a meeting cap c adds +-W(c-L_g) where X_c and Y_{c-L_g} differ.  Uncoupled chains
// (Algorithms 1/2) have (a) only, with w(t) = clamp(t - b + 1, 0, T) and b + T - 1 steps.
//
// The kernel runs (b) and (a) apart.  A slot's pairs run one after the other to their meetings,
// two lanes to a pair (lane i holds X, lane i + 16 holds Y; both take the same draws, so both chains
// are one code path, and the Hamming distance follows the two lanes' flips by ballot).  That fixes
// every C = max(l, tau), and with it how many replications the slot retains.  Then one lane runs X
// again from the start for l steps, once per retained replication: all lanes of a warp take these
// runs in step, so the time, the event weight and part of each Philox block are the warp's, no
// clock is compared, and nothing of Y is in the loop.
// Why apart: in one loop for both, the few unmet lanes of a warp (4.8% of lane-steps, at least one
// in 79% of warp-steps) made every step pay for Y, and the replications of a warp ended one by one.
// Running X's first tau steps twice costs tau / l (5% there).
template <bool COUPLED, bool SYSTEMATIC, bool BATCH, int DEG, bool TRACE = false, bool MARKS = false>
__global__ void __launch_bounds__(pairs_threads(DEG, BATCH), 1) pairs_kernel(const KParams p, const BParams bp) {
    extern __shared__ __align__(16) unsigned char smem[];
    constexpr unsigned FULL = 0xFFFFFFFFu;
    const int warp = threadIdx.x >> 5, lane = threadIdx.x & 31, nwarps = blockDim.x >> 5;
    // Shared memory: [tables (single instance)] [one region per warp].  A region is 32 columns of
    // wpp words, word w of column c at word 32 w + c, so the same byte offset (a row entry) addresses
    // a pool's count in any column and the 32 lanes of a warp touch 32 different banks.
    uint4 *sRows = reinterpret_cast<uint4 *>(smem);
    unsigned long long *sAlias = nullptr, *sT = nullptr;
    int wpp;
    uint32_t *regions;
    if constexpr (!BATCH) {
        sAlias = reinterpret_cast<unsigned long long *>(smem + static_cast<size_t>(p.na) * 16);
        sT = sAlias + p.na;
        for (int i = threadIdx.x; i < p.na; i += blockDim.x) {
            sRows[i] = reinterpret_cast<const uint4 *>(p.rows)[i];
            sAlias[i] = p.alias[i];
        }
        for (int i = threadIdx.x; i < p.nT; i += blockDim.x) sT[i] = p.T[i];
        wpp = p.wpp;
        regions = reinterpret_cast<uint32_t *>(smem + p.smem_tables);
    } else {
        wpp = bp.max_wpp;
        regions = reinterpret_cast<uint32_t *>(smem);
    }
    uint32_t *const st = regions + static_cast<uint32_t>(warp) * 32u * static_cast<uint32_t>(wpp) + lane;  // word w: st[w * 32]
    unsigned char *const cbase = reinterpret_cast<unsigned char *>(st);
    for (int w = 0; w < wpp; ++w) st[w * 32] = 0u;
    if constexpr (!BATCH) st[p.dummy_word_index * 32] = p.dummy_word;
    __syncthreads();

    // This warp's scratch (see warp_words): `bank` entries (a slot's sums, and marks of the clones
    // touched), a list of the entries whose pairs are done, a statistics record per lane, and an entry
    // per pair.
    const int stride_na = BATCH ? bp.max_na : p.na;
    const int bank = BATCH ? bp.bank : p.bank, marks = MARKS ? (BATCH ? bp.marks : p.marks) : 0;
    long long *const wbase = (BATCH ? bp.pair_scratch : p.pair_scratch) +
                             static_cast<size_t>(blockIdx.x * nwarps + warp) *
                                 static_cast<size_t>(warp_words(bank, stride_na, marks, COUPLED));
    const size_t ew = static_cast<size_t>(stride_na) + static_cast<size_t>(marks);
    // Word q of the marks of an entry; word W: events that were not marked.
    auto mark = [&](long long *entry, uint32_t q) { return reinterpret_cast<uint32_t *>(entry + stride_na) + q; };
    auto list = [&]() { return reinterpret_cast<uint32_t *>(wbase + bank * ew); };
    auto pst = [&]() {
        return reinterpret_cast<unsigned long long *>(wbase + bank * ew + bank + lane * kPairStats);
    };
    // Pair i's events of the replication it is running.
    auto pair_sums = [&](int i) { return wbase + bank * ew + bank + 32 * kPairStats + i * ew; };
    unsigned long long *const counters = BATCH ? bp.counters : p.counters;
#pragma unroll
    for (int i = 0; i < kPairStats; ++i) pst()[i] = 0ull;
    auto stat_add = [&](int i, unsigned long long v) { red_add(reinterpret_cast<long long *>(&pst()[i]), static_cast<long long>(v)); };

    // Per-instance values: fixed for a single instance, the chunk's instance in a batch (a chunk
    // never spans two).  Values the steps use live in registers; the others are read where needed.
    const InstDesc *desc = nullptr;
    const uint4 *gRows = nullptr;
    const unsigned long long *gAlias = nullptr, *gT = nullptr;
    int na = 0, deg = 0;
    uint32_t W = 0, ell = 0, instance = 0, k0 = 0, k1 = 0, dummy_entry = 0, ws0 = 0, wcap = 0;
    // A pair marks its events up to this step; one that goes on leaves its slot to be read whole, so that a
    // long one does not pay for a mark per event as well.
    auto marked_steps = [&]() { return static_cast<uint32_t>(na) >> 1; };
#define MCPD_FIELD(name, batch_expr, single_expr) \
    auto name = [&]() { if constexpr (BATCH) return batch_expr; else return single_expr; }
    MCPD_FIELD(v_B, static_cast<uint32_t>(__ldg(&desc->B)), static_cast<uint32_t>(p.B));
    MCPD_FIELD(v_unit, static_cast<uint32_t>(__ldg(&desc->unit)), static_cast<uint32_t>(p.unit));
    MCPD_FIELD(v_step_limit, static_cast<uint32_t>(__ldg(&desc->step_limit)), static_cast<uint32_t>(p.step_limit));
    MCPD_FIELD(v_tau_audit, __ldg(&desc->tau_audit), p.tau_audit);
    MCPD_FIELD(v_capped, __ldg(&desc->capped) != 0, p.capped != 0);
    MCPD_FIELD(v_lag, static_cast<uint32_t>(__ldg(&desc->lag)), static_cast<uint32_t>(p.lag));
    MCPD_FIELD(v_k, __ldg(&desc->k), p.k);
    MCPD_FIELD(v_L, __ldg(&desc->L), p.L);
    MCPD_FIELD(v_burn, __ldg(&desc->burn), p.burn);
    MCPD_FIELD(v_length, __ldg(&desc->length), p.length);
    MCPD_FIELD(v_P, __ldg(&desc->P), p.P);
    MCPD_FIELD(v_slot_offset, __ldg(&desc->slot_offset), p.slot_offset);
    MCPD_FIELD(v_dwi, static_cast<uint32_t>(__ldg(&desc->dummy_word_index)), static_cast<uint32_t>(p.dummy_word_index));
    MCPD_FIELD(v_dw, __ldg(&desc->dummy_word), p.dummy_word);
    MCPD_FIELD(v_wpp, static_cast<uint32_t>(__ldg(&desc->wpp)), static_cast<uint32_t>(p.wpp));
    MCPD_FIELD(v_Tnu, reinterpret_cast<const unsigned long long *>(__ldg(reinterpret_cast<const unsigned long long *>(&desc->Tnu))),
               reinterpret_cast<const unsigned long long *>(p.Tnu));
    MCPD_FIELD(v_init_pairs, reinterpret_cast<const uint32_t *>(__ldg(reinterpret_cast<const unsigned long long *>(&desc->init_pairs))),
               p.init_pairs);
    MCPD_FIELD(v_n_init, __ldg(&desc->n_init_pairs), p.n_init_pairs);
    MCPD_FIELD(v_S1, reinterpret_cast<unsigned long long *>(__ldg(reinterpret_cast<const unsigned long long *>(&desc->S1))), p.S1);
    MCPD_FIELD(v_S2lo, reinterpret_cast<unsigned long long *>(__ldg(reinterpret_cast<const unsigned long long *>(&desc->S2lo))), p.S2lo);
    MCPD_FIELD(v_S2hi, reinterpret_cast<unsigned long long *>(__ldg(reinterpret_cast<const unsigned long long *>(&desc->S2hi))), p.S2hi);
    MCPD_FIELD(v_bcount, reinterpret_cast<unsigned long long *>(__ldg(reinterpret_cast<const unsigned long long *>(&desc->bcount))), p.bcount);
#undef MCPD_FIELD
    auto clamp32 = [](long long v) -> uint32_t { return v < 0 ? 0u : (v > 0xFFFFFFFFll ? 0xFFFFFFFFu : static_cast<uint32_t>(v)); };
    // Rows list a clone's positive-outcome pools first.  Uniform degree 3..kMaskDeg (every clone of
    // the instance, or of every instance of a batched class, sits in exactly DEG pools): their number
    // is the last entry, and thresholds are indexed npos * 64 + (mask of deciding pools).  Other
    // degrees fill all eight entries: the number sits in bits of entry 0 that an offset leaves
    // clear, and n+ and n- are counted from the mask.
    constexpr bool MASKT = DEG >= 3 && DEG <= kMaskDeg;
    auto derive = [&]() {
        ws0 = clamp32(COUPLED ? v_k() : v_burn());
        wcap = clamp32(COUPLED ? v_L() : v_length());
    };
    if constexpr (!BATCH) {
        na = p.na; deg = p.deg; W = p.W;
        dummy_entry = p.dummy_entry;
        ell = static_cast<uint32_t>(COUPLED ? p.ell : p.unit);
        instance = p.instance;
        k0 = static_cast<uint32_t>(p.seed); k1 = static_cast<uint32_t>(p.seed >> 32);
        derive();
    }
    constexpr int NE = DEG > 0 ? DEG : kRow;       // row entries visited per clone
    auto rowAt = [&](uint32_t c) -> uint4 {
        if constexpr (BATCH) return __ldg(gRows + c); else return sRows[c];
    };
    auto aliasAt = [&](uint32_t c) -> unsigned long long {
        if constexpr (BATCH) return __ldg(gAlias + c); else return sAlias[c];
    };
    auto tHi = [&](uint32_t i) -> uint32_t {
        if constexpr (BATCH) return __ldg(reinterpret_cast<const uint32_t *>(gT) + 2 * i + 1);
        else return reinterpret_cast<const uint32_t *>(sT)[2 * i + 1];
    };
    auto tLo = [&](uint32_t i) -> uint32_t {
        if constexpr (BATCH) return __ldg(reinterpret_cast<const uint32_t *>(gT) + 2 * i);
        else return reinterpret_cast<const uint32_t *>(sT)[2 * i];
    };
    auto entries = [&](const uint4 &row, uint32_t *ent) {
        ent[0] = row.x & (MASKT ? 0xFFFFu : 0xFF83u); ent[1] = row.x >> 16; ent[2] = row.y & 0xFFFFu; ent[3] = row.y >> 16;
        ent[4] = row.z & 0xFFFFu; ent[5] = row.z >> 16; ent[6] = row.w & 0xFFFFu; ent[7] = row.w >> 16;
    };
    // Entry l of a row is a real pool (not past the clone's degree, not the padding pool).
    auto real = [&](int l, const uint32_t *ent) -> bool {
        return l < NE && (DEG > 0 || (l < deg && ent[l] != dummy_entry));
    };
    auto wstep = [&](uint32_t u) -> uint32_t { return u < ws0 ? 0u : min(u - ws0 + 1u, wcap); };

    // A lane's state.  role: 0 idle, 1 a single run of X, 2 a pair's X, 3 a pair's Y.
    int role = 0;
    bool on = false;                      // takes steps
    bool dirty = false;                   // some bit of its column may be set
    bool events = false;                  // its pair's sums may hold something
    uint32_t slot_local = 0, slot_g = 0, r = 0, t = 0, S = 0, N = 0, D = 0, stop = 0;
    long long *sum = nullptr;             // where its events go: the slot's entry, or its pair's sums
    int32_t *trec = nullptr;              // TRACE: the record of the current replication
    uint32_t trace_from = 0;              // TRACE: the single run records from its pair's meeting on

    // The site a step word selects (alias draw), and its row, ahead of the step: they depend on the
    // step words only.  Tables in shared memory: one step ahead.  A batch's tables come from L2 (some
    // 300 cycles a load), and the row's address waits for the alias word: the alias word two steps
    // ahead, the row one.
    uint32_t I_cur = 0, col_next = 0, coin_next = 0;
    uint4 row_cur = make_uint4(0u, 0u, 0u, 0u);
    unsigned long long e_next = 0;
    auto column = [&](uint32_t ws) {
        const unsigned long long prod = static_cast<unsigned long long>(ws) * static_cast<uint32_t>(na);
        col_next = static_cast<uint32_t>(prod >> 32);
        coin_next = static_cast<uint32_t>(prod);
        e_next = aliasAt(col_next);
    };
    auto site = [&]() {
        I_cur = coin_next < static_cast<uint32_t>(e_next) ? col_next : static_cast<uint32_t>(e_next >> 32);
        row_cur = rowAt(I_cur);
    };
    auto ahead = [&](uint32_t ws) {       // ws: the site word of the next step, in a batch of the one after
        if constexpr (BATCH) { site(); column(ws); }
        else { column(ws); site(); }
    };
    auto first_site = [&](const uint4 &blk) {
        column(blk.x);
        site();
        if constexpr (BATCH) column(blk.z);
    };

    // One step of one chain: the site's bit z and the counts c of its pools in the lane's column; a
    // pool decides when it holds no other positive (c - z = 0); the threshold the deciding pools
    // select.  The uniform U = wu 2^32 + lo flips the bit if (U < T) != z.  A step loads T's high
    // word and leaves it after one compare unless the bit may flip (`may`); lo is drawn only when wu
    // equals the high word (`flips`).
    struct Site { uint32_t I, q, xw, z, ix, th; uint32_t ent[8], c[kRow]; };
    auto look = [&](Site &s, const uint4 &row) {
        s.q = s.I >> 5;
        s.xw = st[s.q * 32];
        s.z = __funnelshift_r(s.xw, s.xw, s.I) & 1u;
        entries(row, s.ent);
        s.ix = 0;
#pragma unroll
        for (int l = 0; l < kRow; ++l) {
            s.c[l] = 0u;
            if (l < NE && (DEG > 0 || l < deg)) {
                s.c[l] = cbase[s.ent[l]];
                if (s.c[l] == s.z) s.ix |= 1u << l;
            }
        }
        // the threshold's index: of the mask in the positive pools' row, or 9 n+ + n-
        if constexpr (MASKT) s.ix += s.ent[kRow - 1] << 6;
        else s.ix = __popc(s.ix) + 8u * __popc(s.ix & ~(0xFFFFFFFFu << ((row.x >> 2) & 15u)));
        s.th = tHi(s.ix);
    };
    auto may = [&](const Site &s, uint32_t wu) -> bool { return s.z ? wu >= s.th : wu <= s.th; };
    auto flips = [&](const Site &s, uint32_t wu, uint32_t time) -> bool {
        if (wu != s.th) return true;
        const uint32_t lo = philox_low_word(make_uint4(time, r, slot_g, instance | (2u << 24)), k0, k1);
        return (lo < tLo(s.ix) ? 1u : 0u) != s.z;
    };
    // Flip the site's bit and move the counts of its pools (from the values loaded this step).
    auto apply = [&](const Site &s) {
        st[s.q * 32] = s.xw ^ (1u << (s.I & 31));
        const uint32_t delta = s.z ? 0xFFu : 1u;
#pragma unroll
        for (int l = 0; l < kRow; ++l)
            if (real(l, s.ent)) cbase[s.ent[l]] = static_cast<unsigned char>(s.c[l] + delta);
    };
    uint32_t first = 0, cnt = 0;          // the chunk: slots first .. first + cnt - 1

    // Random start Z_0 ~ prod Bernoulli(nu_i) of lane src's new replication, drawn by the whole
    // warp: the lanes take the clone pairs that have some nu_i > 0 (one Philox block each, tag 1, counter
    // (a / 2, r, slot, instance)) and set the bits and pool counts they draw in src's column, and for
    // a pair (X_0 = Y_0) in Y's, with shared-memory atomics (a count word holds four pools of one
    // column, and a count never passes 255, so adding 1 << 8 b touches only its own byte).
    auto coop_init = [&](int src, bool both) {
        const uint32_t r_s = __shfl_sync(FULL, r, src), slot_s = __shfl_sync(FULL, slot_g, src);
        uint32_t *const st_s = st - lane + src;
        unsigned char *const cb_s = reinterpret_cast<unsigned char *>(st_s);
        const unsigned long long *tnu = v_Tnu();
        const uint32_t *ip = v_init_pairs();
        const int n_ip = v_n_init();
        for (int e = lane; e < n_ip; e += 32) {
            const int a = static_cast<int>(__ldg(ip + e));
            const uint4 b = philox10(make_uint4(static_cast<uint32_t>(a) >> 1, r_s, slot_s, instance | (1u << 24)), k0, k1);
#pragma unroll
            for (int h = 0; h < 2; ++h) {
                const int c = a + h;
                if (c >= na) break;
                const unsigned long long u = h ? ((static_cast<unsigned long long>(b.z) << 32) | b.w)
                                               : ((static_cast<unsigned long long>(b.x) << 32) | b.y);
                if (u < __ldg(tnu + c)) {
                    atomicOr(&st_s[(c >> 5) * 32], 1u << (c & 31));
                    if (both) atomicOr(&st_s[(c >> 5) * 32 + 16], 1u << (c & 31));
                    uint32_t ent[8];
                    entries(rowAt(c), ent);
#pragma unroll
                    for (int l = 0; l < kRow; ++l) {
                        if (!real(l, ent)) continue;
                        const uint32_t off = ent[l], one = 1u << (8u * (off & 3u));
                        uint32_t *const word = reinterpret_cast<uint32_t *>(cb_s + (off & ~3u));
                        atomicAdd(word, one);
                        if (both) atomicAdd(word + 16, one);
                    }
                }
            }
        }
        __syncwarp();
    };
    // Random starts of the new replications of the lanes with `mine` (their columns are empty).
    auto start_random = [&](bool mine) {
        if (v_Tnu() == nullptr) return;
        const unsigned all = __ballot_sync(FULL, mine), pair = __ballot_sync(FULL, mine && role >= 2);
        unsigned m = all & ~(pair & 0xFFFF0000u);
        __syncwarp();
        while (m) {
            const int src = __ffs(m) - 1;
            m &= m - 1;
            coop_init(src, (pair >> src) & 1u);
        }
        if (mine) dirty = true;
    };
    // Empty lane src's column, and for a pair (`both`) Y's, by the whole warp; `w` != 0: first add w
    // for every bit set (the closing term of a single run) to its entry.
    auto coop_clear = [&](int src, bool both, uint32_t w) {
        const uint32_t w_s = __shfl_sync(FULL, w, src);
        long long *const sum_s = reinterpret_cast<long long *>(__shfl_sync(FULL, reinterpret_cast<unsigned long long>(sum), src));
        uint32_t *const st_s = st - lane + src;
        for (uint32_t q = lane, e = v_wpp(); q < e; q += 32) {
            if (q < W && w_s) {
                uint32_t m = st_s[q * 32];
                if (MARKS && m) red_or(mark(sum_s, q), m);
                while (m) {
                    const int b = __ffs(m) - 1;
                    m &= m - 1;
                    red_add(sum_s + q * 32 + b, static_cast<long long>(w_s));
                }
            }
            const uint32_t v = (DEG == 0 && q == v_dwi()) ? v_dw() : 0u;
            st_s[q * 32] = v;
            if (both) st_s[q * 32 + 16] = v;
        }
        __syncwarp();
    };
    auto trace_sum = [&](uint32_t idx, int j, long long g) {
        if constexpr (!BATCH) {
            const uint32_t slot = first + idx;
            if (p.trace_stride > 0 && (slot % p.trace_stride) == 0)
                p.trace_G[(static_cast<long long>(slot) / p.trace_stride) * na + j] = g;
        }
    };
    // Add sum g of clone j of entry `idx` to bucket n - 1 (n = 0: the slot is dropped) and zero it.
    auto move = [&](uint32_t idx, uint32_t n, int j, long long g) {
        if (g == 0) return;
        wbase[static_cast<size_t>(idx) * ew + j] = 0;
        if (!n) return;
        bucket_add(v_S1(), v_S2lo(), v_S2hi(), na, static_cast<int>(n) - 1, j, g);
        trace_sum(idx, j, g);
    };
    // All sums of entry `idx`, by the whole warp: coalesced reads, four in flight a lane.
    auto flush = [&](uint32_t idx, uint32_t n) {
        const long long *const from = wbase + static_cast<size_t>(idx) * ew;
        for (int j0 = lane; j0 < na; j0 += 128) {
            long long g[4];
#pragma unroll
            for (int u = 0; u < 4; ++u) g[u] = j0 + 32 * u < na ? __ldcg(from + j0 + 32 * u) : 0;
#pragma unroll
            for (int u = 0; u < 4; ++u) move(idx, n, j0 + 32 * u, g[u]);
        }
        if (lane == 0 && n) atomicAdd(&v_bcount()[n - 1], 1ull);
    };
    // All sums of entries 0 .. cnt - 1, whose slots all retained n replications (uncoupled chains): a lane
    // adds a clone's sums over the slots and brings the totals to the bucket.  (Slot by slot, every slot's
    // three atomics per clone met all other warps' on the bucket: 4.7 million chains of 32 steps on 64 clones
    // took 13.5 ms against 1.7, 0.9 million of one sweep on 333 clones 2.6 against 1.8.)  For fewer than four
    // slots, whose loads in flight are too few: 81 slots of 2424 clones 481 us this way, 458 one by one.
    auto flush_same = [&](uint32_t n) {
        for (int j = lane; j < na; j += 32) {
            long long s1 = 0;
            unsigned long long lo = 0, hi = 0;
            for (uint32_t at = 0; at < cnt; at += 8) {
                long long g[8];
#pragma unroll
                for (int u = 0; u < 8; ++u) g[u] = at + u < cnt ? __ldcg(wbase + static_cast<size_t>(at + u) * ew + j) : 0;
#pragma unroll
                for (int u = 0; u < 8; ++u) {
                    if (g[u] == 0) continue;
                    wbase[static_cast<size_t>(at + u) * ew + j] = 0;
                    trace_sum(at + u, j, g[u]);
                    s1 += g[u];
                    const unsigned long long a = static_cast<unsigned long long>(g[u] < 0 ? -g[u] : g[u]), sq = a * a;
                    lo += sq;
                    hi += __umul64hi(a, a) + (lo < sq ? 1ull : 0ull);
                }
            }
            if (lo | hi) bucket_add_sums(v_S1(), v_S2lo(), v_S2hi(), na, static_cast<int>(n) - 1, j, s1, lo, hi);
        }
        if (lane == 0) atomicAdd(&v_bcount()[n - 1], static_cast<unsigned long long>(cnt));
    };
    // The marked sums of the list's entries, eight entries at a time: a lane takes the next marked clone of
    // each of four, so that four loads, and then four additions, are in flight (one by one, 80,000 slots of 4
    // steps of 5000 clones took 0.18 to 0.38 ms); an entry with events that were not marked is read whole.
    auto flush_marked = [&](uint32_t entries_done, uint32_t reps_each) {
        constexpr int G = 8;
        for (uint32_t at = 0; at < entries_done; at += G) {
            const bool mine = lane < G && at + lane < entries_done;
            const uint32_t my_idx = !mine ? 0u : COUPLED ? __ldcg(list() + 2 * (at + lane)) : at + lane;
            const uint32_t my_n = !mine ? 0u : COUPLED ? __ldcg(list() + 2 * (at + lane) + 1) : reps_each;
            bool whole = false;
            if constexpr (COUPLED) {
                uint32_t *const my_all = mark(wbase + my_idx * ew, W);
                whole = mine && __ldcg(my_all) != 0u;
                if (whole) *my_all = 0u;
            }
            const unsigned all = __ballot_sync(FULL, whole), here = __ballot_sync(FULL, mine);
            uint32_t idx[G], n[G];
#pragma unroll
            for (int u = 0; u < G; ++u) {
                idx[u] = __shfl_sync(FULL, my_idx, u);
                n[u] = __shfl_sync(FULL, my_n, u);
            }
            for (uint32_t q = lane; q < W; q += 32) {
                uint32_t m[G];
#pragma unroll
                for (int u = 0; u < G; ++u) m[u] = (here >> u) & 1u ? __ldcg(mark(wbase + idx[u] * ew, q)) : 0u;
#pragma unroll
                for (int u = 0; u < G; ++u) {
                    if (m[u]) *mark(wbase + idx[u] * ew, q) = 0u;
                    if ((all >> u) & 1u) m[u] = 0u;
                }
#pragma unroll
                for (int h = 0; h < G; h += 4)
                    while (m[h] | m[h + 1] | m[h + 2] | m[h + 3]) {
                        long long g[4];
                        unsigned long long old[4];
                        uint32_t j[4];
#pragma unroll
                        for (int u = 0; u < 4; ++u) {
                            j[u] = q * 32u + static_cast<uint32_t>(__ffs(m[h + u])) - 1u;
                            g[u] = m[h + u] ? __ldcg(wbase + idx[h + u] * ew + j[u]) : 0;
                            m[h + u] &= m[h + u] - 1u;
                        }
#pragma unroll
                        for (int u = 0; u < 4; ++u) {
                            if (g[u] == 0) continue;
                            wbase[idx[h + u] * ew + j[u]] = 0;
                            if (!n[h + u]) continue;
                            old[u] = bucket_add_low(v_S1(), v_S2lo(), na, static_cast<int>(n[h + u]) - 1, static_cast<int>(j[u]), g[u]);
                            trace_sum(idx[h + u], static_cast<int>(j[u]), g[u]);
                        }
#pragma unroll
                        for (int u = 0; u < 4; ++u)
                            if (g[u] && n[h + u])
                                bucket_add_high(v_S2hi(), na, static_cast<int>(n[h + u]) - 1, static_cast<int>(j[u]), g[u], old[u]);
                    }
            }
            __syncwarp();
            if (COUPLED && mine && !whole && my_n) atomicAdd(&v_bcount()[my_n - 1], 1ull);
#pragma unroll
            for (int u = 0; u < G; ++u)
                if ((all >> u) & 1u) flush(idx[u], n[u]);
        }
        if (!COUPLED && lane == 0) atomicAdd(&v_bcount()[reps_each - 1], static_cast<unsigned long long>(entries_done));
    };
    auto record_slot = [&](uint32_t nstar, long long cost, uint32_t reps) {
        if constexpr (!BATCH) {
            if (p.slot_nstar) {
                p.slot_nstar[slot_local] = static_cast<int32_t>(nstar);
                p.slot_S[slot_local] = cost;
                p.slot_reps[slot_local] = static_cast<int32_t>(reps);
            }
        }
    };
    auto trace_at = [&]() {
        if constexpr (TRACE) {
            trec = nullptr;
            if (slot_local % static_cast<uint32_t>(p.trace_stride) == 0 && r < static_cast<uint32_t>(p.trace_reps))
                trec = p.trace_rec + (static_cast<size_t>(slot_local / static_cast<uint32_t>(p.trace_stride)) *
                                      static_cast<size_t>(p.trace_reps) + r) * (4 + static_cast<size_t>(p.trace_steps));
            trace_from = 0;
            // a single run of a coupled replication: its pair recorded the draws before the meeting
            // (all of them if it was stopped unmet)
            if (COUPLED && role == 1 && trec) {
                const int32_t tau = __ldcg(trec);
                trace_from = tau > 0 ? static_cast<uint32_t>(tau) : 0xFFFFFFFFu;
            }
        }
    };
    auto trace_step = [&](uint32_t I, uint32_t time, bool xf, bool yf) {
        if constexpr (TRACE) {
            if (trec && time >= trace_from && time < static_cast<uint32_t>(p.trace_steps))
                trec[4 + time] = static_cast<int32_t>(I | (xf ? 1u << 16 : 0u) | (yf ? 1u << 17 : 0u));
        }
    };
    // Point the lane at slot `idx` of the chunk and its entry.
    auto entry = [&]() { return wbase + static_cast<size_t>(slot_local - first) * ew; };
    auto take = [&](uint32_t idx) {
        slot_local = first + idx;
        slot_g = static_cast<uint32_t>(v_slot_offset() + static_cast<long long>(slot_local));
        sum = entry();
        r = 0;
    };

    for (bool begin = true;; begin = false) {
        // The next chunk of slots.  The first one is the warp's own number, so that a block's warps
        // start on neighbouring chunks (in a batch mostly one instance, whose tables they share
        // through the L1); the rest from one counter.
        {
            unsigned long long s = blockIdx.x * static_cast<unsigned>(nwarps) + static_cast<unsigned>(warp);
            if (!begin) {
                if (lane == 0) s = atomicAdd(&counters[kWork], 1ull);
                s = __shfl_sync(FULL, s, 0) + static_cast<unsigned long long>(gridDim.x) * static_cast<unsigned>(nwarps);
            }
            if constexpr (!BATCH) {
                const unsigned long long at = s * static_cast<unsigned long long>(p.chunk);
                if (at >= static_cast<unsigned long long>(p.P)) break;
                first = static_cast<uint32_t>(at);
                cnt = static_cast<uint32_t>(min(static_cast<unsigned long long>(p.chunk), static_cast<unsigned long long>(p.P) - at));
            } else {
                if (s >= static_cast<unsigned long long>(bp.total_units)) break;
                const long long u = static_cast<long long>(s);
                int lo = 0, hi = bp.n_inst - 1;             // last instance with unit_begin <= u
                while (lo < hi) {
                    const int mid = (lo + hi + 1) >> 1;
                    if (__ldg(&bp.insts[mid].unit_begin) <= u) lo = mid; else hi = mid - 1;
                }
                if (DEG == 0 && desc) st[v_dwi() * 32] = 0u;    // the old layout's padding pool
                desc = bp.insts + lo;
                const InstDesc &d = *desc;
                gRows = reinterpret_cast<const uint4 *>(MASKT ? d.rows_mask : d.rows);
                gAlias = reinterpret_cast<const unsigned long long *>(d.alias);
                gT = reinterpret_cast<const unsigned long long *>(MASKT ? d.T_mask : d.T);
                na = d.na; deg = d.deg; W = d.W;
                dummy_entry = d.dummy_entry;
                ell = static_cast<uint32_t>(COUPLED ? d.ell : d.unit);
                instance = d.instance;
                k0 = static_cast<uint32_t>(d.seed); k1 = static_cast<uint32_t>(d.seed >> 32);
                derive();
                if (DEG == 0) st[v_dwi() * 32] = v_dw();
                // Phase 1 steps every lane, those that have found no slot too (a chunk of fewer than
                // 16), and a step loads by the site drawn ahead: no site of the last chunk's
                // instance, which may have more clones, is carried over.
                if constexpr (COUPLED) {
                    I_cur = col_next = coin_next = 0u;
                    e_next = 0ull;                      // draws site 0
                    row_cur = rowAt(0u);
                }
                const long long P = v_P(), units = d.units, per = (P + units - 1) / units;
                first = static_cast<uint32_t>((u - d.unit_begin) * per);
                cnt = static_cast<uint32_t>(min(per, P - static_cast<long long>(first)));
            }
        }
        // Single runs, the chunk's (slot, replication) pairs: any lane takes any of them, for a
        // slot's sums take reductions from every lane.  The list holds, per slot whose pairs are done,
        // its entry and N (0: dropped); run_n, run_idx are the head's (read once per slot), hr its next
        // replication.
        uint32_t head = 0, hr = 0, ready = 0, run_n = 0, run_idx = 0;
        uint32_t reps_each = 0;           // uncoupled: every slot's replications (no list)
        role = 0; on = false;
        auto assign_runs = [&]() -> bool {
            bool got = false;
            for (;;) {
                const unsigned idle = __ballot_sync(FULL, role == 0);
                if (!idle) break;
                if (hr == run_n) {
                    if (head == ready) break;
                    run_idx = COUPLED ? __ldcg(list() + 2 * head) : head;
                    run_n = COUPLED ? __ldcg(list() + 2 * head + 1) : reps_each;
                    hr = 0;
                    ++head;
                }
                const uint32_t k = min(run_n - hr, static_cast<uint32_t>(__popc(idle)));
                const uint32_t rank = __popc(idle & ((1u << lane) - 1u));
                if (role == 0 && rank < k) {
                    take(run_idx);
                    r = hr + rank;
                    role = 1;
                    got = true;
                }
                hr += k;
            }
            return got;
        };

        // ---- Phase 1: pairs to their meetings, and single runs on the lanes that are left over.
        if constexpr (COUPLED) {
            const uint32_t lag = v_lag();
            const bool quick = ell <= v_step_limit();   // (else a pair that has met runs into its limit)
            uint32_t taken = 0;           // slots handed to pairs
            uint4 blk = make_uint4(0u, 0u, 0u, 0u), nxt = blk;
            auto draw = [&](uint32_t c0) -> uint4 {
                if constexpr (BATCH) return philox10(make_uint4(c0, r, slot_g, instance), k0, k1);
                else return philox10_rk(make_uint4(c0, r, slot_g, instance), p.rk);
            };
            unsigned pm = 0;              // the lanes that hold pairs
            uint32_t still = 0;           // Y stays at Y_0 before t = L
            auto step = [&](uint32_t ws_next, uint32_t wu) {
                Site s;
                s.I = I_cur;
                const uint4 row = row_cur;
                ahead(ws_next);
                look(s, row);
                bool f = on && t >= still && may(s, wu);
                if (TRACE || __any_sync(FULL, f)) {
                    if (f) {
                        f = flips(s, wu, t);
                        if (f) {
                            apply(s);
                            dirty = true;
                            // The event's weight: w(t) of a single run, W(t - L) of a pair.  With
                            // m = min(u, l) and a = m - k + 1: w(u) = a and
                            // W(u) = a (a + 1) / 2 + (u - m) (l - k + 1) (both 0 before k).
                            const bool single = role == 1;
                            const uint32_t u = single ? t : t - lag, m = min(u, ell);
                            if ((single || t >= lag) && m >= ws0) {
                                const uint32_t a = m - ws0 + 1u;
                                long long w = static_cast<long long>((static_cast<unsigned long long>(a) * (single ? 2u : a + 1u)) >> 1) +
                                              static_cast<long long>(static_cast<unsigned long long>(single ? 0u : u - m) * wcap);
                                if (lag != 1u && !single) w = lag_prefix(u, ws0, ell, lag);
                                red_add(sum + s.I, (s.z != 0) != (role == 3) ? w : -w);
                                if (MARKS && (single || t < marked_steps())) red_or(mark(sum, s.q), 1u << (s.I & 31));
                                events = true;
                            }
                        }
                    }
                    const unsigned fb = __ballot_sync(FULL, f);
                    if (fb & pm) {
                        const unsigned zb = __ballot_sync(FULL, s.z != 0);
                        if (role >= 2) {
                            const int o = lane ^ 16;
                            const uint32_t pz = (zb >> o) & 1u, pf = (fb >> o) & 1u;
                            D += ((s.z ^ (f ? 1u : 0u) ^ pz ^ pf)) - (s.z ^ pz);
                        }
                    }
                    if constexpr (TRACE) {
                        if (on) {
                            if (role == 1) trace_step(s.I, t, f, f);
                            else if (role == 2) trace_step(s.I, t, f, (fb >> (lane | 16)) & 1u);
                        }
                    }
                }
                if (on) {
                    ++t;
                    on = t < stop && !(D == 0 && t >= lag);   // a pair stops where it has met
                }
            };
            bool was_on = false, begin = true;
            for (;;) {
                const bool ended = was_on && !on;
                if (begin || __any_sync(FULL, ended)) {
                    begin = false;
                    __syncwarp();         // the columns as every lane's steps left them
                    bool restart = false, done = false, banked = false, keep = false;
                    uint32_t close = 0;
                    const bool pair_ended = ended && role >= 2;
                    if (ended) {
                        if (role == 1) {
                            close = wstep(ell);
                            done = true;
                        } else {
                            // 1 completed (met, or unmet at the meeting cap), 2 doomed (it cannot end
                            // within B), 3 step limit
                            const uint32_t B = v_B();
                            const bool met = D == 0 && t >= lag;
                            const bool capped = !met && v_capped() && t >= v_step_limit();
                            const int how = met || capped ? 1 : ((r > 0 && t >= B - S) ? 2 : 3);
                            const uint32_t C = met ? max(ell, t) : t, tau = met ? t : 0u;
                            if (TRACE && trec && role == 2) {
                                trec[0] = static_cast<int32_t>(tau);
                                trec[1] = static_cast<int32_t>(C);
                                trec[2] = how;
                                trec[3] = static_cast<int32_t>(r);
                            }
                            bool over = false;             // the slot ends here
                            keep = how == 1;
                            if (keep) {
                                if (capped && role == 2) {     // the open intervals of X_c and Y_{c-L}
                                    const long long wc = t < lag ? 0ll : lag_prefix(t - lag, ws0, ell, lag);
                                    for (uint32_t q = 0; q < W && wc != 0; ++q) {
                                        const uint32_t xw = st[q * 32];
                                        uint32_t dm = xw ^ st[q * 32 + 16];
                                        if (!dm) continue;
                                        if (MARKS) red_or(mark(entry(), q), dm);
                                        while (dm) {
                                            const int b = __ffs(dm) - 1;
                                            dm &= dm - 1;
                                            red_add(entry() + q * 32 + b, ((xw >> b) & 1u) ? wc : -wc);
                                        }
                                    }
                                }
                                S += C;
                                N += 1;
                                if (role == 2) {
                                    stat_add(kPsSumTau, tau);
                                    red_max(&pst()[kPsMaxTau], tau);
                                    const long long audit = v_tau_audit();
                                    if (audit > 0 && (tau > audit || tau == 0u)) stat_add(kPsTauAudit, 1);
                                    if (S > B) stat_add(kPsZero, 1);   // only a slot's first replication ends beyond B
                                }
                                if (S < B && B - S >= v_unit()) { ++r; restart = true; } else over = true;
                            } else {
                                over = true;
                            }
                            if (over) {
                                if (role == 2) {
                                    // draws: the retained replications' and the stopped one's
                                    const unsigned long long prog = static_cast<unsigned long long>(S) + (how == 1 ? 0u : t);
                                    const unsigned long long reps = r + 1ull;
                                    stat_add(kPsProgress, prog);
                                    stat_add(kPsStarted, reps);
                                    stat_add(kPsRetained, N);
                                    stat_add(kPsSiteUpdates, 2 * prog - reps * lag);
                                    if (how == 2) stat_add(kPsAborted, 1);
                                    if (how == 3) {
                                        stat_add(kPsLimit, 1);
                                        atomicExch(BATCH ? bp.error : p.error, 1);
                                    }
                                    if (how == 3) N = 0;          // the slot is dropped
                                    record_slot(N, static_cast<long long>(S), r + 1);
                                    banked = true;
                                }
                                done = true;
                            }
                        }
                    }
                    // A retained replication's events join its slot's sums; those of a doomed one, or of
                    // a pair at its step limit, go.  Coalesced, by the whole warp; pairs that met before
                    // the window have none.
                    {
                        unsigned m = __ballot_sync(FULL, pair_ended && events);
                        m = (m | m >> 16) & 0xFFFFu;
                        if (m) {
                            __threadfence();
                            __syncwarp();
                            while (m) {
                                const int src = __ffs(m) - 1;
                                m &= m - 1;
                                const bool keep_s = __shfl_sync(FULL, keep ? 1 : 0, src) != 0;
                                long long *const to = wbase + static_cast<size_t>(__shfl_sync(FULL, slot_local, src) - first) * ew;
                                long long *const from = pair_sums(src);
                                bool all = true;
                                if constexpr (MARKS) {
                                    all = __shfl_sync(FULL, t, src) > marked_steps();
                                    for (uint32_t q = lane; q < W; q += 32) {
                                        uint32_t b = __ldcg(mark(from, q));
                                        if (!b) continue;
                                        *mark(from, q) = 0u;
                                        if (keep_s) red_or(mark(to, q), b);
                                        while (!all && b) {
                                            const uint32_t j = q * 32 + __ffs(b) - 1;
                                            b &= b - 1;
                                            const long long g = __ldcg(from + j);
                                            from[j] = 0;
                                            if (keep_s) red_add(to + j, g);
                                        }
                                    }
                                    if (all && keep_s && lane == 0) red_or(mark(to, W), 1u);
                                }
                                for (int j0 = all ? lane : na; j0 < na; j0 += 128) {
                                    long long g[4];
#pragma unroll
                                    for (int u = 0; u < 4; ++u) g[u] = j0 + 32 * u < na ? __ldcg(from + j0 + 32 * u) : 0;
#pragma unroll
                                    for (int u = 0; u < 4; ++u)
                                        if (g[u] != 0) {
                                            from[j0 + 32 * u] = 0;
                                            if (keep_s) red_add(to + j0 + 32 * u, g[u]);
                                        }
                                }
                            }
                            __threadfence();
                            __syncwarp();
                            if (pair_ended) events = false;
                        }
                    }
                    // columns of the ended lanes (where nothing flipped they are empty)
                    {
                        const unsigned pair = __ballot_sync(FULL, pair_ended && dirty);
                        unsigned m = __ballot_sync(FULL, ended && role == 1 && dirty) | ((pair | pair >> 16) & 0xFFFFu);
                        __syncwarp();
                        while (m) {
                            const int src = __ffs(m) - 1;
                            m &= m - 1;
                            coop_clear(src, ((pair | pair >> 16) >> src) & 1u, close);
                        }
                        if (ended) dirty = false;
                    }
                    // a slot whose pairs are done goes on the list
                    {
                        const unsigned m = __ballot_sync(FULL, banked);
                        if (banked) {
                            const uint32_t at = ready + __popc(m & ((1u << lane) - 1u));
                            list()[2 * at] = slot_local - first;
                            list()[2 * at + 1] = N;
                        }
                        ready += __popc(m);
                        __syncwarp();
                        if (done) role = 0;
                    }
                    // free lanes: pairs for the slots that are left, then single runs
                    if (taken < cnt) {
                        const unsigned idle = __ballot_sync(FULL, role == 0);
                        const unsigned pairs = idle & (idle >> 16) & 0xFFFFu;
                        const uint32_t me = static_cast<uint32_t>(lane) & 15u;
                        const uint32_t at = taken + __popc(pairs & ((1u << me) - 1u));
                        if (((pairs >> me) & 1u) && at < cnt) {
                            role = lane < 16 ? 2 : 3;
                            take(at);
                            sum = pair_sums(lane & 15);
                            S = 0; N = 0;
                            restart = true;
                        }
                        taken = min(cnt, taken + __popc(pairs));
                    }
                    pm = __ballot_sync(FULL, role >= 2);
                    if (taken == cnt && pm != 0 && ell > 0 && assign_runs()) restart = true;
                    start_random(restart);
                    if (restart) {
                        t = 0;
                        // Only a pair's Hamming distance comes to 0: a single run stops at l, and
                        // so does a pair if its step limit lies below l (it runs into the limit).
                        D = role == 1 || !quick ? 0x40000000u : 0u;
                        still = role == 3 ? lag : 0u;
                        stop = role == 1 ? ell : min(r > 0 ? v_B() - S : 0xFFFFFFFFu, v_step_limit());
                        trace_at();
                        on = true;
                        blk = draw(0);
                        if constexpr (BATCH) nxt = draw(1);
                        first_site(blk);
                    }
                    if (!__any_sync(FULL, on)) break;
                }
                was_on = on;
                if constexpr (BATCH) {
                    const uint4 after = draw((t >> 1) + 2);
                    step(nxt.x, blk.y);
                    step(nxt.z, blk.w);
                    blk = nxt;
                    nxt = after;
                } else {
                    nxt = draw((t >> 1) + 1);
                    step(blk.z, blk.y);
                    step(nxt.x, blk.w);
                    blk = nxt;
                }
            }
        } else {
            const uint32_t B = v_B(), n = max(1u, B / ell);      // ell: a chain's b + T - 1 >= 1 steps
            for (uint32_t idx = lane; idx < cnt; idx += 32) {
                take(idx);
                stat_add(kPsProgress, static_cast<unsigned long long>(n) * ell);
                stat_add(kPsSiteUpdates, static_cast<unsigned long long>(n) * ell);
                stat_add(kPsStarted, n);
                stat_add(kPsRetained, n);
                if (ell > B) stat_add(kPsZero, 1);
                record_slot(n, static_cast<long long>(n) * ell, n);
            }
            ready = cnt;
            reps_each = n;
        }

        // ---- Phase 2: single runs, all lanes in step.
        for (;;) {
            assign_runs();
            if (!__any_sync(FULL, role == 1)) break;
            start_random(role == 1);
            if (role == 1) {
                trace_at();
                // Rounds 1 and 2 of the Philox blocks (c0, r, slot, instance): the products of slot and
                // r are fixed for the replication, those of c0 and instance are the warp's.
                const uint32_t rk0 = BATCH ? k0 : p.rk[0];
                const uint32_t sl = kPhiloxM1 * slot_g;
                const uint32_t a1 = __umulhi(kPhiloxM1, slot_g) ^ r ^ rk0;
                const uint32_t h2 = __umulhi(kPhiloxM0, a1), l2 = kPhiloxM0 * a1;
                auto draw = [&](uint32_t c0) -> uint4 {
                    const uint32_t h0 = __umulhi(kPhiloxM0, c0), l0 = kPhiloxM0 * c0;
                    const uint32_t z1 = h0 ^ instance ^ (BATCH ? k1 : p.rk[1]);
                    const uint32_t hz = __umulhi(kPhiloxM1, z1), lz = kPhiloxM1 * z1;
                    if constexpr (BATCH) {
                        const uint32_t a0 = k0 + kPhiloxW0, b0 = k1 + kPhiloxW1;
                        return philox_tail(make_uint4(hz ^ sl ^ a0, lz, h2 ^ l0 ^ b0, l2), a0 + kPhiloxW0, b0 + kPhiloxW1);
                    } else {
                        return philox_tail_rk(make_uint4(hz ^ sl ^ p.rk[2], lz, h2 ^ l0 ^ p.rk[3], l2), p.rk);
                    }
                };
                uint32_t sysI = 0;
                auto step = [&](uint32_t ws_next, uint32_t wu, uint32_t time) {
                    Site s;
                    uint4 row;
                    if (SYSTEMATIC) {
                        s.I = sysI;
                        row = rowAt(sysI);
                        ++sysI;
                        if (sysI == static_cast<uint32_t>(na)) sysI = 0;
                    } else {
                        s.I = I_cur;
                        row = row_cur;
                        ahead(ws_next);
                    }
                    look(s, row);
                    const bool m = may(s, wu);
                    if (TRACE || m) {
                        const bool f = m && flips(s, wu, time);
                        trace_step(s.I, time, f, COUPLED && f);
                        if (f) {
                            apply(s);
                            const uint32_t w = wstep(time);
                            if (w) {
                                red_add(sum + s.I, s.z ? static_cast<long long>(w) : -static_cast<long long>(w));
                                if (MARKS) red_or(mark(sum, s.q), 1u << (s.I & 31));
                            }
                        }
                    }
                };
                uint4 blk = draw(0);
                if (!SYSTEMATIC) first_site(blk);
                uint32_t time = 0;
                // both steps of a block inlined, the next block drawn between them
                if constexpr (BATCH) {
                    uint4 nxt = draw(1);
                    for (; time + 2 <= ell; time += 2) {
                        step(nxt.x, blk.y, time);
                        const uint4 after = draw((time >> 1) + 2);
                        step(nxt.z, blk.w, time + 1);
                        blk = nxt;
                        nxt = after;
                    }
                } else {
                    for (; time + 2 <= ell; time += 2) {
                        step(blk.z, blk.y, time);
                        const uint4 nxt = draw((time >> 1) + 1);
                        step(nxt.x, blk.w, time + 1);
                        blk = nxt;
                    }
                }
                if (ell & 1u) step(blk.z, blk.y, time);
                // The closing terms w(l) of X_l's bits, and the column back to empty: every lane its
                // own, together.
                const uint32_t w = wstep(ell);
                for (uint32_t q = 0; q < W; ++q) {
                    const uint32_t xw = st[q * 32];
                    if (xw) {
                        st[q * 32] = 0u;
                        uint32_t m = w ? xw : 0u;
                        if (MARKS && m) red_or(mark(sum, q), m);
                        while (m) {
                            const int b = __ffs(m) - 1;
                            m &= m - 1;
                            red_add(sum + q * 32 + b, static_cast<long long>(w));
                        }
                    }
                }
                for (uint32_t q = W, e = v_wpp(); q < e; ++q) st[q * 32] = (DEG == 0 && q == v_dwi()) ? v_dw() : 0u;
                dirty = false;
                if (TRACE && !COUPLED && trec) {
                    trec[0] = 0;
                    trec[1] = static_cast<int32_t>(ell);
                    trec[2] = 1;
                    trec[3] = static_cast<int32_t>(r);
                }
            }
            __syncwarp();
            role = 0;
        }

        // ---- The chunk's sums to their buckets: every lane's reductions into the entries are performed
        // before they are read, and the zeros before the next chunk reduces into them.
        __threadfence();
        __syncwarp();
        if constexpr (MARKS) flush_marked(ready, reps_each);
        else if (!COUPLED && cnt >= 4) flush_same(reps_each);
        else if constexpr (!COUPLED) for (uint32_t at = 0; at < cnt; ++at) flush(at, reps_each);
        else for (uint32_t at = 0; at < ready; ++at) flush(__ldcg(list() + 2 * at), __ldcg(list() + 2 * at + 1));
        __threadfence();
        __syncwarp();
    }

    // Every lane of the warp is here: sum (or max) the lanes' statistics over the warp.
    const int dst[kPairStats] = {kProgress, kRepsStarted, kRepsRetained, kRepsAborted,
                                 kZeroCompletion, kStepLimitHits, kSumTau, kMaxTau, kTauOverAudit,
                                 kSiteUpdates};
    __threadfence();
#pragma unroll
    for (int i = 0; i < kPairStats; ++i) {
        unsigned long long v = __ldcg(&pst()[i]);
        for (int o = 16; o > 0; o >>= 1) {
            const unsigned long long u = __shfl_down_sync(FULL, v, o);
            v = i == kPsMaxTau ? max(v, u) : v + u;
        }
        if (lane == 0 && v) {
            if (i == kPsMaxTau) atomicMax(&counters[dst[i]], v);
            else atomicAdd(&counters[dst[i]], v);
        }
    }
}

}  // namespace
}  // namespace mcpd
