// Sizes that the kernels and the host's plans share.  No CUDA.
#pragma once

namespace wc {

constexpr int kHeadDim = 128;
constexpr int kPage = 16;
constexpr int kBands = 8;
constexpr int kMaxGroup = 8;

// Per (query head, split) partial: acc[128] | m | l | D | Tier-B D | value
// term | max ||v|| | pad.  140 floats: in the CTA merge's shared buffer the
// rows of the heads one warp instruction touches then start in distinct bank
// groups (12 words apart modulo 32; 136 would put two heads on each group).
constexpr int kPartialStride = kHeadDim + 12;

// Page streams per decode CTA: warps (fp8), or producer / consumer warp pairs.
constexpr int kPageStreams = 8, kG32PageStreams = 6;

}  // namespace wc
