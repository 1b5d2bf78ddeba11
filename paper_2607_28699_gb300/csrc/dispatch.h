// Which variant of a kernel a call takes: rules on its sizes, types and alignment alone, each
// with both sides measured on GB300.  Host code only, no CUDA.
#pragma once

#include <cstdint>

#include "../../include/witcert.h"

namespace wc {

// ---- repair selection: threads per cell -----------------------------------------------------
// A wide CTA has fewer positions a thread and ends sooner, a narrow one needs fewer warps and
// barriers per cell; the wide one wins while the cells' threads take at most half of the
// chip's (152 SMs of 2048).  Us wide / narrow: 128 pages, 280 cells 3.4 / 4.1, 2800 7.4 / 6.8;
// 256 pages, 280 3.8 / 4.3, 784 5.8 / 5.2; 1000 pages, 112 5.1 / 6.0, 784 14.7 / 13.4; 4096
// pages, 28 11.3 / 12.0, 280 21.2 / 16.7.
constexpr bool repair_wide(int64_t cells, int threads) { return cells * threads <= 152 * 1024; }

}  // namespace wc
