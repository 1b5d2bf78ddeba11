// Which variant of a kernel a call takes: rules on its sizes, types and alignment alone, each
// with both sides measured on GB300.  Host code only, no CUDA.
#pragma once

#include <cstdint>

#include "../../include/witcert.h"

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
// 8192 6.3 / 5.3, 32768 15.2 / 9.3; 4096 rows, 8 heads 5.5 / 5.3, 16 6.6 / 8.6, 32 6.9 / 12.7;
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

}  // namespace wc
