// Constants and helpers shared by the decode kernels (fragment layouts of
// mma.sync m16n8k16 / m16n8k8 and the exact int8 / dither -> fp16 operands).
#pragma once

#include <cuda.h>

#include <climits>

#include "wc_kernels.cuh"

namespace wc {

namespace {

// Extra outputs compiled into a decode kernel (template bit mask).
constexpr int kXTierB = 1;   // Tier-B meter (§4.2)
constexpr int kXValue = 2;   // value-side witness terms and output bound (§3, §4.2)
constexpr int kXRepair = 4;  // per-page meter terms for block-level repair selection (§6.3.5)
constexpr int kXAppend = 8;  // the decode writes the step's new token before reading it
constexpr int kXFlat = 16;   // warp-specialized kernel under the flattened split plan
// failure-detection test (warp-specialized kernel, split plan): one page's
// copies are never issued and every wait gives up after kStallTries tries
constexpr int kXStall = 32;
constexpr int kStallTries = 64;
constexpr float kLog2e = 1.4426950408889634f;
constexpr float kRsd = 0.08838834764831845f;                      // 1/sqrt(128)
constexpr float kRsdLog2e = 0.08838834764831845f * 1.4426950408889634f;

constexpr uint32_t kSel01 = 0x4140u, kSel23 = 0x4342u;   // [x0,K,x1,K], [x2,K,x3,K]

__device__ __forceinline__ uint32_t sel_interleave(int p) {  // [a_p, b_p, a_p+1, b_p+1]
    return p == 0 ? 0x5140u : 0x7362u;
}

template <int kBits>
struct DitherConst;
template <>
struct DitherConst<8> {  // xi = (j + 1/2)/256 - 1/2 = h' - kappa, h' = 4 + j/256
    static constexpr float kappa = 4.498046875f;
};
template <>
struct DitherConst<10> {  // xi = (j + 1/2)/1024 - 1/2 = h' - kappa, h' = 1 + j/1024
    static constexpr float kappa = 1.49951171875f;
};

// h' pair (fp16) for two 8-bit dithers: bytes of x at the selector.
__device__ __forceinline__ uint32_t h8(uint32_t x, uint32_t sel) { return prmt(x, 0x44444444u, sel); }
// -h' pair (fp16) for two 8-bit dithers: the same bytes under a negative high byte.
__device__ __forceinline__ uint32_t nh8(uint32_t x, uint32_t sel) { return prmt(x, 0xC4C4C4C4u, sel); }
// h' pair (fp16) for two 10-bit dithers in the low bits of each 16-bit lane.
__device__ __forceinline__ uint32_t h10(uint32_t x) { return (x & 0x03FF03FFu) | 0x3C003C00u; }

// Upward margin on the merged e-form accumulator D = E_p~[e^c - 1] (and the
// Tier-B one) before the meter (A^2 - 1)/2 = D (D + 2)/2 is formed, so the
// fp32 meter lands on or above the exact value of §3 Thm. "Sound replacement"
// instead of within rounding either side of it.  It covers:
//  - ex2.approx near 1 (relative error below 2^-22 of 2^c, i.e. an absolute
//    error below 2^-22 in each e^c - 1 and so in their p~-weighted mean): kDAbs;
//  - the fp32 sums of p~ and p~ (e^c - 1) (per lane about a thousand terms
//    at 32k tokens, then the warp, CTA and split merges: n u < 2^-13), the
//    hi + lo fp16 bound operand (2^-22) and the rounding of the logits that
//    move p~ (their effect on D, measured against the fp64 oracle, stays near
//    10^-5 relative): kDRel, at about 4x the larger of these.
// At 1 + 2^-12 it stays well inside the 1e-3 relative parity tolerance.
constexpr float kDRel = 1.0f + 0x1p-12f;
constexpr float kDAbs = 0x1p-21f;
__device__ __forceinline__ float d_upper(float d) { return fmaf(d, kDRel, kDAbs); }

// One token's meter term p~ (e^c - 1) in the log2 frame of the running maximum:
// t = y - m (p~ = 2^t, flushed to 0 below 2^-126) and cl = c log2(e).  The
// kernels use the product 2^t (2^cl - 1) as long as every cl of the page is below
// kHugeLog2: an underflowed 2^t then drops less than 2^(64 - 126) per token,
// far inside kDAbs.  A page with a larger bound (a key row of huge magnitude;
// never with ordinary inputs) takes its terms from meter_term, which uses
// 2^(t + cl) from kHugeLog2 on, its exponent raised by a bound on the two fp32
// roundings of t + cl + margin: at least the term, and finite wherever the term
// is, so a token whose weight underflows but whose bound does not still counts
// (the product gives 0, or 0 * inf = NaN).
constexpr float kHugeLog2 = 64.0f;
__device__ __forceinline__ float meter_term(float t, float cl) {
    if (cl < kHugeLog2) return fast_exp2(t) * (fast_exp2(cl) - 1.f);
    if (t == -INFINITY) return 0.f;   // a token past the context
    return fast_exp2(t + cl + (fabsf(t) + cl) * 0x1p-22f);
}

// NaN only arises in the meter from 0 * inf or inf - inf, i.e. from a term or a
// sum that overflowed: report it as +inf, the bound's overflow value.
__device__ __forceinline__ float raw_or_inf(float raw) { return raw == raw ? raw : INFINITY; }

// 2^n for -126 <= n <= 127.
__device__ __forceinline__ float pow2(int n) { return __int_as_float((127 + n) << 23); }

// Two bytes of w_xor80 (code ^ 0x80) at the selector as 1152 + code - sub, exact.
__device__ __forceinline__ uint32_t u8x2_minus(uint32_t w_xor80, uint32_t sel, uint32_t sub) {
    const uint32_t h = prmt(w_xor80, 0x64646464u, sel);
    const __half2 v = __hsub2(*reinterpret_cast<const __half2*>(&h), *reinterpret_cast<const __half2*>(&sub));
    return *reinterpret_cast<const uint32_t*>(&v);
}

__device__ __forceinline__ uint32_t word_of(const uint4& v, int i) {
    return i == 0 ? v.x : i == 1 ? v.y : i == 2 ? v.z : v.w;
}

// Transpose of an 8x8 b16 matrix held in the mma fragment layout.
__device__ __forceinline__ uint32_t movmatrix_t(uint32_t x) {
    uint32_t y;
    asm volatile("movmatrix.sync.aligned.m8n8.trans.b16 %0, %1;" : "=r"(y) : "r"(x));
    return y;
}

// Token held by row r of a 16-row QK / softmax tile in the warp-specialized
// decode: rows 2i, 2i+1 hold tokens 4i, 4i+1 and rows 8+2i, 9+2i tokens
// 4i+2, 4i+3, so the P fragment transposed by movmatrix gives lane (g, c) the
// tokens 4c .. 4c+3 that ldmatrix.trans delivers for V.
__device__ __forceinline__ int tok_row(int r) { return 4 * ((r & 7) >> 1) + 2 * (r >> 3) + (r & 1); }

// ldmatrix.trans of two 16x16 byte blocks: lanes 0-15 address the 16 rows of
// the first, lanes 16-31 those of the second; lane (g, c) receives, per block,
// column g (first word) and column g + 8 (second word) at rows 4c .. 4c+3.
__device__ __forceinline__ void ldsm_t_b8_x2(uint32_t (&d)[4], const void* row) {
    asm volatile("ldmatrix.sync.aligned.m16n16.x2.trans.shared.b8 {%0, %1, %2, %3}, [%4];"
                 : "=r"(d[0]), "=r"(d[1]), "=r"(d[2]), "=r"(d[3])
                 : "r"(smem_addr(row)));
}

// ldmatrix.trans of four 8x8 blocks of 16-bit elements: lanes 8i .. 8i+7 address
// block i's rows; lane (g, c) receives, per block, column g at rows 2c, 2c+1.
__device__ __forceinline__ void ldsm_t_b16_x4(uint32_t (&d)[4], const void* row) {
    asm volatile("ldmatrix.sync.aligned.m8n8.x4.trans.shared.b16 {%0, %1, %2, %3}, [%4];"
                 : "=r"(d[0]), "=r"(d[1]), "=r"(d[2]), "=r"(d[3])
                 : "r"(smem_addr(row)));
}

// Byte offset of 16-byte chunk q of token row t in a tile written with the
// 128-byte swizzle (tile 1024-byte aligned): chunk q of row t sits at chunk
// q ^ (t & 7), so the 8 rows a warp touches per instruction hit distinct banks.
__device__ __forceinline__ int swz(int t, int q) { return t * kHeadDim + 16 * (q ^ (t & 7)); }

__device__ __forceinline__ void tma_page(void* dst, const CUtensorMap* map, int z, uint64_t* bar) {
    asm volatile(
        "cp.async.bulk.tensor.3d.shared::cluster.global.tile.mbarrier::complete_tx::bytes [%0], [%1, {%2, %3, %4}], "
        "[%5];" ::"r"(smem_addr(dst)),
        "l"(reinterpret_cast<uint64_t>(map)), "r"(0), "r"(0), "r"(z), "r"(smem_addr(bar))
        : "memory");
}

// Fetches a tensor map ahead of its first copy.
__device__ __forceinline__ void prefetch_map(const CUtensorMap* map) {
    asm volatile("prefetch.tensormap [%0];" ::"l"(reinterpret_cast<uint64_t>(map)) : "memory");
}

// A CTA's work as segments: pages [a, e) of unit (b, h); page stream (warp
// pair) w of the CTA's n takes pages a + ((w - ph) mod n) + n i.  Split plan: one segment, the
// CTA's split (possibly empty).  Flattened plan: CTA c serves KV head
// h = c mod Hkv and takes share j = c / Hkv of the batch laid end to
// end (sequence after sequence), cut at sequence boundaries; the Hkv CTAs of a
// share read the same pages together (the heads of a page are adjacent in the
// cache).  A segment costs its pages and a fixed part (query setup, the CTA's merge, the
// streams' last round), so in the layout kCutPages empty positions follow every sequence
// with pages but the last: a share that goes on to a next sequence gets that many pages
// less.  The shares start half of that before multiples of their length, so that
// nearly equal sequences, one to a share, are not cut for a page or two.  4 KV heads, us a
// decode: 2 sequences of 987 and 989 pages 21.7 without empty positions and 19.8 with 12
// (what two take that end with a share), 16 of 280 to 512 pages 45.3 and 43.3 (with 8:
// 43.9), 38 of 51 and 53 pages 20.0 (22.1 with shares from 0).
// ph keeps the streams' round robin running across the cuts, so
// every stream gets ceil or floor of the share's pages / n.
constexpr uint32_t kCutPages = 12;

struct WsSeg {
    int b, h, a, e, ph, ctx, np;
    uint32_t vb, hi;   // flattened plan: sequence b's first position; the share's end
};

// Positions of a sequence of np pages in the flattened layout, and positions of a share.
__device__ __forceinline__ uint32_t flat_span(uint32_t np) { return np > 0 ? np + kCutPages : 0u; }
struct FlatShares {
    uint32_t total;   // positions, without the empty ones behind the last sequence
    uint32_t R, off;  // share j: positions [j R - off, (j + 1) R - off); off < R, so share 0 has pages if any has
    __device__ __forceinline__ FlatShares(uint32_t spans, uint32_t shares) {   // spans: sum of flat_span
        total = spans - min(spans, kCutPages);
        off = min(kCutPages / 2, max(1u, (total + shares - 1) / shares) - 1);
        R = max(1u, (total + off + shares - 1) / shares);
    }
};

__device__ __forceinline__ int clamped_ctx(const DecodeParams& p, int b) {
    return max(0, min(load_dep(p.ctx_lens + b), p.max_pages * kPage));
}

// The split plan's segment of this CTA.
__device__ __forceinline__ void split_segment(const DecodeParams& p, WsSeg& sg) {
    sg.b = blockIdx.z;
    sg.h = blockIdx.y;
    int ctx = load_dep(p.ctx_lens + sg.b);
    if (ctx < 0 || ctx > p.max_pages * kPage) {
        if (threadIdx.x == 0 && blockIdx.x == 0 && sg.h == 0) atomicOr(p.status, WC_DEV_BAD_CTX);
        ctx = max(0, min(ctx, p.max_pages * kPage));
    }
    sg.ctx = ctx;
    sg.np = (ctx + kPage - 1) / kPage;
    sg.a = blockIdx.x * p.pages_per_split;
    sg.e = min(sg.a + p.pages_per_split, sg.np);
    sg.ph = 0;
    sg.vb = sg.hi = 0;
}

// First segment of the flattened plan; called by every thread of the CTA (a scan of the
// batch's page counts with two block barriers).  cx: this thread's context length, when the
// batch has at most a sequence per thread.  False: no pages.  All positions fit
// in 32 bits (the plan's condition on batch * max_pages, and kCutPages more a sequence).
struct FlatScratch {
    uint32_t wtot[32];
    int b, a, ctx;
    uint32_t vb;
};
__device__ __forceinline__ bool flat_first_segment(const DecodeParams& p, WsSeg& sg, FlatScratch& s, int cx, bool& bad) {
    const int nt = blockDim.x, t = threadIdx.x, per = (p.batch + nt - 1) / nt, cap = p.max_pages * kPage;
    auto length = [&](int i) { return per == 1 ? cx : load_dep(p.ctx_lens + t * per + i); };
    uint32_t loc = 0;
    bad = false;
    for (int i = 0; i < per; ++i)
        if (t * per + i < p.batch) {
            const int len = length(i);
            bad |= len < 0 || len > cap;
            loc += flat_span((uint32_t)(max(0, min(len, cap)) + kPage - 1) / kPage);
        }
    uint32_t inc = loc;   // inclusive scan over the warp
#pragma unroll
    for (int o = 1; o < 32; o <<= 1) {
        const uint32_t v = __shfl_up_sync(0xffffffffu, inc, o);
        if ((t & 31) >= o) inc += v;
    }
    if ((t & 31) == 31) s.wtot[t >> 5] = inc;
    if (t == 0) s.b = -1;
    __syncthreads();
    uint32_t before = 0, total = 0;
    for (int w = 0; w < nt / 32; ++w) {
        const uint32_t v = s.wtot[w];
        total += v;
        if (w < (t >> 5)) before += v;
    }
    const uint32_t excl = before + inc - loc;   // positions of the sequences before this thread's
    const uint32_t hk = p.num_kv_heads, shares = max(1u, p.splits / hk);
    const FlatShares f(total, shares);
    const uint32_t j = (uint32_t)blockIdx.x / hk, lo = max(j * f.R, f.off) - f.off, hi = min(f.total, (j + 1) * f.R - f.off);
    if (lo < hi && excl <= lo + kCutPages && lo < excl + loc) {   // the first page at lo or behind it
        uint32_t vb = excl;
        for (int i = 0; i < per && t * per + i < p.batch; ++i) {
            const int len = max(0, min(length(i), cap));
            const uint32_t np = (uint32_t)(len + kPage - 1) / kPage;
            if (np > 0 && vb <= lo + kCutPages && lo < vb + np) {   // one sequence at most
                s.b = t * per + i;
                s.a = lo > vb ? (int)(lo - vb) : 0;
                s.ctx = len;
                s.vb = vb;
                break;
            }
            vb += flat_span(np);
        }
    }
    __syncthreads();
    if (s.b < 0 || hi <= s.vb) return false;   // the share lies in empty positions
    sg.b = s.b;
    sg.a = s.a;
    sg.h = (int)((uint32_t)blockIdx.x % hk);
    sg.ctx = s.ctx;
    sg.vb = s.vb;
    sg.hi = hi;
    sg.np = (sg.ctx + kPage - 1) / kPage;
    sg.e = (int)min((uint32_t)sg.np, hi - sg.vb);
    sg.ph = 0;
    return true;
}

// Next segment of the flattened plan (the next sequence with pages); false
// at the end of the CTA's share.
template <int kStreams>
__device__ __forceinline__ bool ws_next_segment(const DecodeParams& p, WsSeg& sg) {
    const int done = sg.ph + (sg.e - sg.a);
    do {   // sequences without pages hold no part of the share
        sg.vb += flat_span(sg.np);
        if (sg.vb >= sg.hi || sg.b + 1 >= p.batch) return false;
        ++sg.b;
        sg.ctx = clamped_ctx(p, sg.b);
        sg.np = (sg.ctx + kPage - 1) / kPage;
    } while (sg.np == 0);
    sg.a = 0;
    sg.e = (int)min((uint32_t)sg.np, sg.hi - sg.vb);
    sg.ph = done % kStreams;
    return true;
}

// The flattened plan's first segment, before and after the grid-dependency wait.  While the
// preceding kernel drains, the plan is made of the context lengths as they stand and
// warm() may prefetch what it says (hints: read past L1, clamped into range).  After the wait the lengths
// are read again, and the plan is made anew if one has changed.  bad: a length is out of range.
template <typename Warm>
__device__ __forceinline__ bool flat_plan(const DecodeParams& p, WsSeg& sg, FlatScratch& s, Warm warm) {
    const bool single = p.batch <= (int)blockDim.x, mine = single && (int)threadIdx.x < p.batch;
    int cx = mine ? __ldcg(p.ctx_lens + threadIdx.x) : 0;
    bool waited = false, have, bad;
    for (;;) {
        if (!single && !waited) {
            grid_dep_wait();
            waited = true;
        }
        have = flat_first_segment(p, sg, s, cx, bad);
        if (waited) break;
        if (have) warm(sg);
        grid_dep_wait();
        waited = true;
        const int now = mine ? load_dep(p.ctx_lens + threadIdx.x) : 0;
        const bool changed = now != cx;
        cx = now;
        if (!__syncthreads_or(changed)) break;
    }
    if (bad && blockIdx.x == 0) atomicOr(p.status, WC_DEV_BAD_CTX);
    return have;
}

// While the preceding kernel drains: a page's codes, scales and witnesses into L2.  The
// page-table entry may still be changing, so it serves as an address only (clamped).
__device__ __forceinline__ void warm_page(const DecodeParams& p, int b, int h, int lp, int scale_bytes) {
    const int phys = min(max(__ldcg(p.block_table + (size_t)b * p.max_pages + lp), 0), p.num_pages - 1);
    const size_t z = (size_t)phys * p.num_kv_heads + h;
    bulk_prefetch_l2(p.k_codes + z * (kPage * kHeadDim), kPage * kHeadDim);
    bulk_prefetch_l2(p.v_codes + z * (kPage * kHeadDim), kPage * kHeadDim);
    bulk_prefetch_l2(reinterpret_cast<const uint8_t*>(p.k_scale) + z * scale_bytes, scale_bytes);
    bulk_prefetch_l2(reinterpret_cast<const uint8_t*>(p.v_scale) + z * scale_bytes, scale_bytes);
    bulk_prefetch_l2(p.k_witness + z * (kPage * kBands), kPage * kBands * 2);
}
__device__ __forceinline__ void warm_queries(const DecodeParams& p, int b, int h) {
    bulk_prefetch_l2(p.q + ((size_t)b * p.num_q_heads + (size_t)h * p.group) * kHeadDim, p.group * kHeadDim * 2);
}

// Flattened plan: each warp's walker lives in a shared slot, so that only the
// current segment's indices take registers in the page loop; lane 0 advances it.
template <int kStreams>
__device__ __forceinline__ bool ws_step(const DecodeParams& p, WsSeg* slot, int lane) {
    __syncwarp();
    int more = 0;
    if (lane == 0) more = ws_next_segment<kStreams>(p, *slot);
    __syncwarp();
    return __shfl_sync(0xffffffffu, more, 0) != 0;
}

template <int kStreams>
__device__ __forceinline__ int ws_seg_pages(const WsSeg& sg, int w, int& first) {
    first = sg.a + (int)((unsigned)(w - sg.ph + kStreams) % kStreams);
    return first < sg.e ? (sg.e - first + kStreams - 1) / kStreams : 0;
}

}  // namespace

// One layer's code array [num_pages][Hkv][16][128] bytes as a 3-D tensor map
// (channel, slot, page * Hkv + head) whose box is one page of one head,
// written to shared memory with the 128-byte swizzle (swz above).
bool encode_page_map(CUtensorMap* map, const void* codes, int num_pages, int num_kv_heads);

// The split-K merge for the extra outputs in the bit mask x (0, kXTierB,
// kXValue or kXRepair), launched as a programmatic dependent of the decode.
cudaError_t launch_merge_x(const DecodeParams& p, int x, cudaStream_t stream);

}  // namespace wc
