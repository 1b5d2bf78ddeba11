// Which variant of a kernel a call takes: rules on its sizes, types and alignment alone, each
// with both sides measured on GB300.  Host code only, no CUDA.
#pragma once

#include <algorithm>
#include <cstddef>
#include <cstdint>

#include "../../include/witcert.h"
#include "sizes.h"

namespace wc {

// ---- write: one or two tasks (rows of 4 units) per warp -------------------------------------
// From this many tokens on the grid runs per KV head.
constexpr int kPerHeadMinTokens = 16;

// Two: the K and the V rows of the same units in one warp.  The grouped row routine is the
// longest: until its two-task CTAs fill the SMs (6 x 152 of 16 units), one task per warp is
// done sooner (tokens x 8 heads, us one / two tasks: 100 3.8 / 4.5, 600 5.2 / 6.7, 1200 6.8 /
// 8.5).  With the 10-bit dither's two Philox calls a row it is while the one-task CTAs fit the
// SMs at once (7 x 152 of 8 units; one / two tasks, several writes in a row: 64 2.9 / 3.5, 512
// 3.9 / 5.4, 1000 4.6 / 6.2; a write by itself: 1000 6.3 / 7.0, 1500 8.1 / 7.6).
constexpr int64_t kGroupedTwoTaskUnits = 16384, kTenBitTwoTaskUnits = 7 * 152 * 8 + 1;
constexpr bool write_two_tasks(int scheme, int bits, int64_t n_tok, int64_t num_kv_heads) {
    return n_tok >= kPerHeadMinTokens &&
           (scheme == WC_SCHEME_DITHER_INT8_G32             ? n_tok * num_kv_heads >= kGroupedTwoTaskUnits
            : scheme == WC_SCHEME_DITHER_INT8 && bits == 10 ? n_tok * num_kv_heads >= kTenBitTwoTaskUnits
                                                            : true);
}

// ---- pair selection: a cluster of 16 CTAs per KV head, or of 8 ------------------------------
// The wide cluster's copies are 16 bytes; it is launched while every head's cluster is resident
// at once (resident: the device's answer for that launch, 14 on GB300; 0 where 16 CTAs cannot be
// placed).  Heads, us narrow / wide: 4 heads, 1024 rows 3.8 / 4.6, 2048 4.5 / 4.6, 4096 4.8 / 4.4,
// 8192 6.3 / 5.3, 32768 14.9 / 8.7; 4096 rows, 8 heads 5.5 / 5.3, 16 6.6 / 8.6, 32 6.9 / 12.7;
// 65536 rows, 8 heads 46.0 / 26.6, 16 55.3 / 52.3, 32 79.9 / 93.5.
constexpr int kWidePairRows = 4096;
constexpr bool pairs_wide(int n_tok, bool aligned16, int num_kv_heads, int resident) {
    return n_tok >= kWidePairRows && aligned16 && num_kv_heads <= resident;
}

// ---- repair selection: threads per cell -----------------------------------------------------
// A wide CTA has fewer positions a thread and ends sooner, a narrow one needs fewer warps and
// barriers per cell; the wide one wins while the cells' threads take at most half of the
// chip's (152 SMs of 2048).  Us wide / narrow: 128 pages, 280 cells 3.4 / 4.1, 2800 7.4 / 6.8;
// 256 pages, 280 3.8 / 4.3, 784 5.8 / 5.2; 1000 pages, 112 5.1 / 6.0, 784 14.7 / 13.4; 4096
// pages, 28 11.3 / 12.0, 280 21.2 / 16.7.
constexpr bool repair_wide(int64_t cells, int threads) { return cells * threads <= 152 * 1024; }

// ---- decode: how the pages are cut ----------------------------------------------------------
// Workspace layout (bytes): [0, 256) status word, then the partials
// (256-byte aligned).
struct DecodePlan {
    int splits;            // flattened plan: the grid's CTAs
    int pages_per_split;   // 0: the flattened plan
    bool two_per_sm;       // 10-bit dither: the kernel with two CTAs per SM (split plan)
    size_t partials_off, total;
};

// Split plan.  A CTA's n page streams each take every n-th page of its split,
// so a split of P pages costs ceil(P / n) page steps, and a wave of resident
// CTAs adds a fixed prologue / epilogue of about one and a half page steps.
// The split count minimises
//     waves * (ceil(pages_per_split / n) + 1.5),   waves = ceil(CTAs / resident CTAs),
// so a grid never spills a small remainder into an extra wave; splits keep at
// least n pages (one per stream).  Ties go to fewer splits (less to merge).
inline long split_pages(long units, int max_pages, long slots, long streams) {
    constexpr long kWaveCost2 = 3;    // per-wave fixed cost, in half page steps
    const long max_splits = std::max<long>(1, std::min<long>(max_pages / streams, 4 * slots));
    long best_pps = std::max(max_pages, 1), best_cost = -1;
    for (long sp = 1; sp <= max_splits; ++sp) {
        const long pps = (max_pages + sp - 1) / sp;
        const long splits = (max_pages + pps - 1) / pps;
        if (splits != sp) continue;   // same plan as a smaller split count
        const long waves = (splits * units + slots - 1) / slots;
        const long cost = waves * (2 * ((pps + streams - 1) / streams) + kWaveCost2);
        if (best_cost < 0 || cost < best_cost) {
            best_cost = cost;
            best_pps = pps;
        }
    }
    return best_pps;
}

// A batch with block tables of at most kShortRounds rounds of pages takes the split plan: a share
// of the flattened one would have a cut every few rounds.  4 KV heads of 7 query heads, us
// split / flattened: 32 sequences of 4 pages 6.9 / 9.4, 16 of 5 to 19 8.3 / 10.3, 32 of 4 to 31 12.0 /
// 13.3; 8 KV heads, 32 of 8 to 60 30.4 / 28.3.
// With the 8-bit dither the flattened plan is the faster one all the same where a unit's split
// CTA costs much beside its cut: over several waves with few query heads per KV head
// (less to merge at a cut), and with the append over more than one wave.  5 pages, 8 KV heads,
// split / flattened: 76 sequences of 1 query head each 19.4 / 18.1, of 3 20.7 / 20.1, of 8 26.9 / 28.2;
// 200 of 1 48.1 / 38.5, of 5 59.0 / 54.1; append, 2 to 5 pages: 32 of 4 14.8 / 13.9, 200 of 8 83.2 / 68.5.
constexpr long kShortRounds = 5;
constexpr bool short_table_flat(long units, int num_sms, int scheme, int bits, int group, bool append) {
    return scheme == WC_SCHEME_DITHER_INT8 && bits == 8 &&
           (append ? units > num_sms : units >= 4L * num_sms && group <= (units >= 10L * num_sms ? 5 : 3));
}

// The 10-bit dither has two kernels: warp pairs, one CTA per SM (a page's dither is drawn beside
// the consuming warp), and two CTAs of 8 warps per SM (drawn by the warp itself: slower pages, but
// one CTA's prologue and merge under the other's pages).  The second is the faster one where its
// CTAs fill the SMs (units >= 2 x 152) with tables so short that a unit's fixed part counts, on
// the split plan: a CTA starts when another ends, which evens out lengths while the tables are a
// small part of an SM's work.  us, pairs / two per SM, equal lengths | a quarter of the table
// and up | one long sequence among short ones:
//   38 sequences x 8 KV heads, 20 pages 24.3 / 21.5 | 24.2 / 21.3 | 17.9 / 16.7, 40 36.7 / 34.4 | 33.5 / 31.7 | 20.4 / 24.6
//   76 x 8, 41 pages 73.4 / 66.8 | 53.8 / 55.1 | 29.9 / 26.8, 60 95.2 / 91.2 | 75.0 / 81.1 | 35.0 / 33.9
//   300 x 4, 80 pages 250 / 231 | 185 / 176 | 79.5 / 60.8, 120 352 / 332 | 249 / 250 | 95.0 / 76.0
//   1000 x 4, 5 pages 195 / 127 | 176 / 117 | 169 / 103
constexpr long kTwoPerSmPages = 24;   // of the table, per unit that an SM's two CTAs each take
constexpr bool ten_bit_two_per_sm(long units, int max_pages, int num_sms) {
    const long slots2 = 2L * num_sms;
    return units >= slots2 && max_pages * slots2 <= kTwoPerSmPages * units;
}

// available: the workspace's bytes (a smaller plan is taken where the preferred one does
// not fit and calls with that size have always been accepted); SIZE_MAX: the preferred plan.
// The size does not depend on group and append.
inline DecodePlan plan_decode(int batch, int num_kv_heads, int max_pages, int num_sms, int scheme, int bits, int group,
                              bool append, size_t available = SIZE_MAX) {
    DecodePlan pl;
    const long units = (long)batch * num_kv_heads;
    // Resident CTAs per SM: the dithered kernels take a whole SM, the fp8 kernel two CTAs.
    const long slots = std::max<long>(1, (long)num_sms * (scheme == WC_SCHEME_FP8_E4M3 ? 2 : 1));
    const long streams = scheme == WC_SCHEME_DITHER_INT8_G32 ? kG32PageStreams : kPageStreams;
    const long best_pps = split_pages(units, max_pages, slots, streams);
    pl.two_per_sm = false;
    pl.pages_per_split = (int)best_pps;
    pl.splits = (int)std::max<long>(1, (max_pages + best_pps - 1) / best_pps);
    long partials = units * pl.splits;
    // A batch of several sequences (lengths unknown to the host, often ragged)
    // takes the flattened plan on the dithered caches: Hkv x floor(SMs / Hkv)
    // CTAs, all resident, each taking a share of one KV head's pages.  fp8
    // keeps the split plan: its CTAs are scheduled as SMs free up, which already
    // evens out a ragged batch, and its pages are cheap.
    const bool batched = batch > 1 && (long long)batch * max_pages < (1LL << 31) && scheme != WC_SCHEME_FP8_E4M3;
    const bool short_table =
        max_pages <= kShortRounds * streams && !short_table_flat(units, num_sms, scheme, bits, group, append);
    const int shares = std::max(1, (int)(slots / num_kv_heads));
    const long flat_partials = (long)num_kv_heads * shares + units;
    auto bytes = [](long n) {
        return (256 + sizeof(float) * (size_t)n * kMaxGroup * kPartialStride + 255) & ~(size_t)255;
    };
    bool flat = batched;
    if (scheme == WC_SCHEME_DITHER_INT8 && bits == 10) {
        // The 10-bit dither's workspace is at least the size it was first given, for two
        // CTAs per SM (and, on a batch that left some empty, a partial per warp of eight).
        // The flattened plan of a batch whose units fill two CTAs per SM with a split each
        // needs up to a partial per SM more: in a workspace of the first size, and beyond
        // the allocation-free call's limit, such a batch takes the two CTAs per SM.
        const long slots2 = std::max<long>(1, 2L * num_sms), pps2 = split_pages(units, max_pages, slots2, 8);
        const long splits2 = std::max<long>(1, (max_pages + pps2 - 1) / pps2);
        long first = units * splits2;
        if (batched && first < slots2) first = 8L * num_kv_heads * std::max<long>(1, slots2 / num_kv_heads) + units;
        if (short_table && partials <= first) flat = false;
        const long most = flat ? std::max(first, flat_partials) : first;   // the workspace of either kernel
        pl.two_per_sm = ten_bit_two_per_sm(units, max_pages, num_sms) ||
                        (flat ? most > first && bytes(most) > available : partials > first);
        if (pl.two_per_sm) {
            flat = false;
            pl.pages_per_split = (int)pps2;
            pl.splits = (int)splits2;
        }
        partials = bytes(most) <= available ? most : first;
    } else if (batched) {
        if (short_table && partials <= flat_partials) flat = false;
        partials = flat_partials;   // the workspace of either
    }
    if (flat) {
        pl.splits = num_kv_heads * shares;
        pl.pages_per_split = 0;
    }
    pl.partials_off = 256;
    pl.total = bytes(partials);
    return pl;
}

}  // namespace wc
