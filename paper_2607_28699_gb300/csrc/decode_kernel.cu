// Metered decode attention (§6 meter loop, read path; §6.2.1-§6.2.2):
// dequantize the paged cache, compute the compressed attention output, and in
// the same pass accumulate the Tier-A e-form meter
//   c_t = (1/sqrt d) sum_b ||q_b|| w_{t,b}        (Thm. "Sound black-box logit bound")
//   A   = sum_t p~_t e^{c_t},  meter = min(1, (A^2 - 1)/2)   (Thm. "Sound replacement")
// merged across context splits under log-sum-exp weights (A is a p~-weighted
// mean, so it merges exactly like the output; §6.2.2).
//
// Two kernels.  decode_kernel (fp8-e4m3, and the 10-bit dither's batches of many short
// sequences): grid (splits, Hkv, batch), 8 warps per
// CTA, two CTAs per SM; each warp owns a 3-stage ring of page buffers in shared
// memory that one of its lanes fills ahead of use: the K and V code tiles (2 KiB
// each) by tensor-map TMA with the 128-byte swizzle (so the 16-byte reads of a warp
// phase hit distinct banks), the witness by a bulk copy, all completing on the
// stage's mbarrier; a page is 16 tokens of one KV head.  Warps run independently
// until the CTA's closing merge.  decode_ws_kernel (dithered INT8, 8-bit and 10-bit
// dither): below.
//
// Per page a warp computes, on mma.sync (fp16 in, fp32 accumulate):
//   QK:    S[token][head]  = code . q - h' . q                m16n8k16, A = codes / dither
//   bound: C[token][head]  = W[token][band] . a[band][head]    m16n8k16, a = ||q_b||/sqrt(d), hi and lo along k
//   PV:    acc[dim][head] += V^T P^T - H^T P^T                 m16n8k16, B = P^T (hi + lo, movmatrix)
// Integer codes and the dither enter the tensor cores as exact fp16 values
// (h' = 4 + j/256 for 8-bit, 1 + j/1024 for 10-bit dither; xi = h' - kappa),
// so code - xi = code - h' + kappa is carried exactly to the fp32 accumulators.
//
// What bounds the pages, measured on GB300 (mixes of instructions in registers, per
// SM sub-partition): an mma.sync m16n8k16 takes 8.1 cycles and keeps its
// sub-partition from issuing for about 7 of them (with four PRMT or FFMA beside it
// 11-12); IMAD.WIDE takes 4 and about 2 of the ALU port (with two LOP3 beside it
// 6.6-7.8); beside an mma.sync it costs 6.  So instructions count, not one pipe.
#include <cuda.h>
#include <cudaTypedefs.h>

#include <climits>

#include "decode_common.cuh"
#include "write_row.cuh"

namespace wc {

namespace {

constexpr int kWarps = 8;
constexpr int kThreads = 32 * kWarps;
constexpr int kStages = 3;
constexpr int kMinBlocks = 2;            // two CTAs (16 warps) per SM
constexpr int kStageBytes = 4416;        // copy bytes: K codes | V codes | K scale | V scale | witness
// Shared memory: the K and V code tiles of every (warp, stage), [16][128] bytes
// each, written by tensor-map TMA with the 128-byte swizzle (1024-byte aligned
// regions), then each stage's scales and witness, then the barriers.
constexpr int kTileRegion = kWarps * kStages * 2048;
constexpr int kOffKs = 0, kOffVs = 32, kOffW = 64;   // within a stage's small part
constexpr int kOffVw = 320;              // value witness [16][2] fp16 (value side)
constexpr int kSmallStride = 384;
constexpr int kOffQ = 2 * kTileRegion + kWarps * kStages * kSmallStride + kWarps * kStages * 8;   // query fragment (kQShared)
constexpr int kQBytes = 16 * 32 * 4;
// Only the variants that use the query fragment's 2 KiB have them (fp8, value side, 300 pages
// x 4 heads: 7.60 us a decode without them, 7.95 with them).
template <bool kInt8, int kX>
struct TwoPerSm {
    static constexpr bool kQShared = kInt8 && (kX & (kXTierB | kXValue)) != 0;
    static constexpr int kSmemBytes = kOffQ + (kQShared ? kQBytes : 0) + 1024;
    static_assert(kOffQ % 16 == 0 && 2 * (kSmemBytes + 1024) <= 228 * 1024, "two CTAs per SM");
};

// decode_kernel's parameters: the code tiles' tensor maps and the call.
struct DkParams {
    CUtensorMap k_map;   // k_codes as [num_pages * Hkv][16][128] bytes, box = one page of one head
    CUtensorMap v_map;
    DecodeParams p;
};

// §6.3.5 "Block-level paging": the share of D of logical page lp for this
// thread's softmax heads 2c, 2c+1, kept against the running maximum it was
// summed under; with the final (M, L) the page contributes d 2^(m - M) / L.
// dpg holds the thread's tokens g, g+8 on entry; the sum runs over the rows g.
__device__ __forceinline__ void emit_page_terms(const DecodeParams& p, int b, int h, int G, int lp, int g, int c,
                                                float (&dpg)[2], const float (&m_run)[2]) {
#pragma unroll
    for (int o = 4; o < 32; o <<= 1) {
        dpg[0] += __shfl_xor_sync(0xffffffffu, dpg[0], o);
        dpg[1] += __shfl_xor_sync(0xffffffffu, dpg[1], o);
    }
    if (g == 0) {
        float2* dst = p.page_terms + ((size_t)b * p.num_q_heads + (size_t)h * G) * p.max_pages + lp;
        if (2 * c < G) dst[(size_t)(2 * c) * p.max_pages] = make_float2(m_run[0], dpg[0]);
        if (2 * c + 1 < G) dst[(size_t)(2 * c + 1) * p.max_pages] = make_float2(m_run[1], dpg[1]);
    }
}

// A page the kernel could not read (outside the pool) contributes nothing.
__device__ __forceinline__ void emit_skipped_page(const DecodeParams& p, int b, int h, int G, int lp, int lane) {
    if (lane < G)
        p.page_terms[((size_t)b * p.num_q_heads + (size_t)h * G + lane) * p.max_pages + lp] =
            make_float2(-INFINITY, 0.f);
}

// q fragment of the B operand (head g, channels 32c + 2i, +1 in word i).
__device__ __forceinline__ void load_q_frag(const DecodeParams& p, int b, int h, int G, int g, int c,
                                            uint32_t (&qw)[16]) {
    const bool row_valid = g < G;
    const uint4* qsrc = reinterpret_cast<const uint4*>(
        p.q + ((size_t)b * p.num_q_heads + (size_t)h * G + (row_valid ? g : 0)) * kHeadDim + 32 * c);
#pragma unroll
    for (int i = 0; i < 4; ++i) {
        const uint4 v = row_valid ? load_dep(qsrc + i) : make_uint4(0, 0, 0, 0);
        qw[4 * i] = v.x; qw[4 * i + 1] = v.y; qw[4 * i + 2] = v.z; qw[4 * i + 3] = v.w;
    }
}

// kInt8: the dithered INT8 cache with the 10-bit dither; otherwise fp8-e4m3.
template <bool kInt8, int kX>
__global__ void __launch_bounds__(kThreads, kMinBlocks) decode_kernel(const __grid_constant__ DkParams dp) {
    constexpr bool kTierB = (kX & kXTierB) != 0, kValue = (kX & kXValue) != 0, kRepair = (kX & kXRepair) != 0;
    static_assert(kInt8 || !kTierB, "Tier B needs the dither");
    const DecodeParams& p = dp.p;
    extern __shared__ __align__(1024) uint8_t smem_raw[];
    uint8_t* smem = smem_raw + ((1024 - (smem_addr(smem_raw) & 1023)) & 1023);
    const int lane = threadIdx.x & 31, warp = threadIdx.x >> 5;
    const int g = lane >> 2, c = lane & 3;
    const int split = blockIdx.x, h = blockIdx.y, b = blockIdx.z;
    const int G = p.group;

    uint8_t* my_k = smem + warp * kStages * 2048;   // this warp's K code tiles; its V tiles kTileRegion on
    uint8_t* my_small = smem + 2 * kTileRegion + warp * kStages * kSmallStride;
    uint64_t* bars =
        reinterpret_cast<uint64_t*>(smem + 2 * kTileRegion + kWarps * kStages * kSmallStride) + warp * kStages;
    if (lane == 0)
        for (int s = 0; s < kStages; ++s) mbar_init(&bars[s], 1);
    fence_barrier_init();
    // the dependent merge may be scheduled now: it waits for this whole grid
    // (griddepcontrol.wait) and launches only once every CTA here has started
    grid_dep_launch();
    grid_dep_wait();   // q, page tables and the cache may come from the preceding kernel

    const bool row_valid = g < G;
    const int p0 = split * p.pages_per_split;
    const int32_t* bt_row = p.block_table + (size_t)b * p.max_pages;
    // Independent loads first: context length, this warp's first page-table
    // entries and the query fragments do not depend on one another.
    int ring[kStages];   // physical pages of this warp's next kStages pages
    uint32_t qw[16];     // head g, channels 32c + 2i, +1 in word i
    const int lim = min(p0 + p.pages_per_split, p.max_pages);
#pragma unroll
    for (int k = 0; k < kStages; ++k) {
        const int lp = p0 + warp + kWarps * k;
        ring[k] = lp < lim ? load_dep(bt_row + lp) : -1;
    }
    int ctx = load_dep(p.ctx_lens + b);
    load_q_frag(p, b, h, G, g, c, qw);
    // Tier B and the value side of the dithered cache read the query fragment (the same in every
    // warp) from shared memory page by page: with its 16 registers held through the PV products
    // they spill (3% of a call; the plain and the repair variant do not gain).
    constexpr bool kQShared = TwoPerSm<kInt8, kX>::kQShared;
    uint4* q_s = reinterpret_cast<uint4*>(smem + kOffQ) + lane;
    if constexpr (kQShared) {
        if (warp == 0) {
#pragma unroll
            for (int i = 0; i < 4; ++i) q_s[32 * i] = make_uint4(qw[4 * i], qw[4 * i + 1], qw[4 * i + 2], qw[4 * i + 3]);
        }
        __syncthreads();
    }
    if (ctx < 0 || ctx > p.max_pages * kPage) {
        if (threadIdx.x == 0 && split == 0 && h == 0) atomicOr(p.status, WC_DEV_BAD_CTX);
        ctx = max(0, min(ctx, p.max_pages * kPage));
    }
    const int npages = (ctx + kPage - 1) / kPage;
    const int p1 = min(p0 + p.pages_per_split, npages);
    const int n_my = (p1 - p0 - warp > 0) ? (p1 - p0 - warp + kWarps - 1) / kWarps : 0;

    // ---- per-warp stage ring --------------------------------------------------
    auto issue = [&](int k, int phys) {   // by one elected lane: the copies' operands stay on the uniform path
        if (k >= n_my || !elect_one()) return;
        uint64_t* bar = &bars[k % kStages];
        if (phys < 0 || phys >= p.num_pages) {
            atomicOr(p.status, WC_DEV_BAD_PAGE);
            asm volatile("mbarrier.arrive.shared::cta.b64 _, [%0];" ::"r"(smem_addr(bar)) : "memory");
            return;
        }
        const int s = k % kStages;
        uint8_t* st = my_small + s * kSmallStride;
        const int z = phys * p.num_kv_heads + h;
        const size_t ph = (size_t)z;
        mbar_arrive_expect_tx(bar, (kInt8 ? kStageBytes : 2048 + 2048 + 256) + (kValue ? 64 : 0));
        tma_page(my_k + s * 2048, &dp.k_map, z, bar);
        tma_page(my_k + kTileRegion + s * 2048, &dp.v_map, z, bar);
        if constexpr (kInt8) {
            bulk_g2s(st + kOffKs, p.k_scale + ph * kPage, 32, bar);
            bulk_g2s(st + kOffVs, p.v_scale + ph * kPage, 32, bar);
        }
        bulk_g2s(st + kOffW, p.k_witness + ph * (kPage * kBands), 256, bar);
        if constexpr (kValue) bulk_g2s(st + kOffVw, p.v_witness + ph * (kPage * 2), 64, bar);
    };
    __syncwarp();
#pragma unroll
    for (int k = 0; k < kStages; ++k) {
        issue(k, ring[k]);
        __syncwarp();
    }

    // ---- band norms and the bound operand ----------------------------------------
    uint32_t a_hi = 0, a_lo = 0;   // B operand of the bound: a[head g][bands 2c, 2c+1]
    float alpha0 = 0.f, alpha1 = 0.f, zoff0 = 0.f, zoff1 = 0.f;   // of the softmax heads 2c, 2c+1
    constexpr float kKappa = DitherConst<10>::kappa;
    constexpr uint32_t kSubV = 0x647F647Fu;                       // 1152 - 1 (u8x2_minus)
    {
        float part[4] = {0.f, 0.f, 0.f, 0.f}, qsum = 0.f;
#pragma unroll
        for (int i = 0; i < 16; ++i) {
            const float2 f = __half22float2(*reinterpret_cast<const __half2*>(&qw[i]));
            if constexpr (kInt8) qsum += f.x + f.y;
            part[i >> 2] = fmaf(f.x, f.x, fmaf(f.y, f.y, part[i >> 2]));   // channels 32c + 8(i>>2) .. +7
        }
        if constexpr (kInt8) {   // kappa * sum(q)
            qsum += __shfl_xor_sync(0xffffffffu, qsum, 1);
            qsum += __shfl_xor_sync(0xffffffffu, qsum, 2);
            zoff0 = kKappa * __shfl_sync(0xffffffffu, qsum, 8 * c);
            zoff1 = kKappa * __shfl_sync(0xffffffffu, qsum, 8 * c + 4);
        }
        if constexpr (kTierB) {   // §4.2: u_t = alpha s_t with alpha = sqrt(2 log(2S/delta) ||q||^2 / (12 d))
            float qn2 = part[0] + part[1] + part[2] + part[3];   // ||q_g||^2 over channels 32c .. 32c+31
            qn2 += __shfl_xor_sync(0xffffffffu, qn2, 1);
            qn2 += __shfl_xor_sync(0xffffffffu, qn2, 2);
            const float lg = p.tb_log_2_over_delta + logf((float)max(ctx, 1));   // log(2S / delta)
            const float al = sqrtf(2.0f * lg * qn2 * (1.0f / (12.0f * kHeadDim)));
            alpha0 = __shfl_sync(0xffffffffu, al, 8 * c);
            alpha1 = __shfl_sync(0xffffffffu, al, 8 * c + 4);
        }
        float band_a, band_b;   // squared norms of bands 2c and 2c+1 of head g
        if (p.rope_layout == WC_ROPE_HALF) {
            // lane c holds the first (c < 2) or second (c >= 2) halves of bands 4(c&1) + i
#pragma unroll
            for (int i = 0; i < 4; ++i) part[i] += __shfl_xor_sync(0xffffffffu, part[i], 2);
            const int src = (lane & ~3) | (c >> 1);
            float v[4];
#pragma unroll
            for (int i = 0; i < 4; ++i) v[i] = __shfl_sync(0xffffffffu, part[i], src);
            band_a = (c & 1) ? v[2] : v[0];
            band_b = (c & 1) ? v[3] : v[1];
        } else {
            band_a = part[0] + part[1];   // dims 32c .. 32c+15 = band 2c
            band_b = part[2] + part[3];
        }
        if (row_valid) {
            const float x0 = sqrtf(band_a) * kRsd, x1 = sqrtf(band_b) * kRsd;
            const __half h0 = __float2half_rn(x0), h1 = __float2half_rn(x1);
            a_hi = pack_h2(__half2float(h0), __half2float(h1));
            a_lo = pack_h2(x0 - __half2float(h0), x1 - __half2float(h1));
        }
    }

    // ---- running state (heads 2c, 2c+1) ----------------------------------------------
    // Log2-domain softmax reference, moved lazily: only when a page's max
    // exceeds it by more than 8 (P may reach 2^8 in between).
    float m_run[2] = {-INFINITY, -INFINITY};
    float l_part[2] = {0.f, 0.f}, d_part[2] = {0.f, 0.f};
    float vt_part[2] = {0.f, 0.f};   // value side: sum p~ rho^v (kValue)
    float vmax = 0.f;                // value side: max ||v|| over this thread's tokens
    float acc[8][4];
#pragma unroll
    for (int i = 0; i < 8; ++i) acc[i][0] = acc[i][1] = acc[i][2] = acc[i][3] = 0.f;
    float db_part[2] = {0.f, 0.f};   // Tier-B meter (kTierB)
    float spv_part[2] = {0.f, 0.f};  // sum P s_v (kInt8)
    // P * s_v * 2^lam_exp stays below 2^14 (fp16): s_v * 2^lam_exp < 2^6 (fp8: s_v = 1).  It only
    // decreases; sv_lim = 2^(6 - lam_exp) is the scale at which it must, FLT_MIN until the
    // first positive scale.
    int lam_exp = kInt8 ? INT_MIN : 6;
    float sv_lim = 1.17549435e-38f;
    const uint32_t c1 = (uint32_t)p.layer * 65536u + (uint32_t)h;   // Philox counter word (kInt8)
    bool failed = false;
    int consumed = 0;

    for (int k = 0; k < n_my; ++k) {
        const int lp = p0 + warp + kWarps * k;   // this page
        // the page-table entry of the page issued at the end of the iteration
        const int phys_issue = (k + kStages < n_my) ? load_dep(bt_row + lp + kWarps * kStages) : -1;
        const int phys = ring[0];
        const bool page_ok = phys >= 0 && phys < p.num_pages;
        const bool landed = mbar_wait_bounded(&bars[k % kStages], (uint32_t)((k / kStages) & 1));
        if (!__all_sync(0xffffffffu, landed)) {   // warp-uniform decision
            if (lane == 0) atomicOr(p.status, WC_DEV_TIMEOUT);
            failed = true;
            break;
        }
        consumed = k + 1;
        if (page_ok) {
            const uint8_t* st = my_small + (k % kStages) * kSmallStride;
            const uint8_t* kt = my_k + (k % kStages) * 2048;   // V tile at kt + kTileRegion
            const int nvalid = min(kPage, ctx - lp * kPage);

            // ---------------- QK: S[token][head] --------------------------------
            // rows g and g+8 are tokens g and g+8; dc[0..3] =
            // (tok g, head 2c), (tok g, 2c+1), (tok g+8, 2c), (tok g+8, 2c+1)
            float dc[4] = {0.f, 0.f, 0.f, 0.f};
            if constexpr (kQShared) {
#pragma unroll
                for (int i = 0; i < 4; ++i) {
                    const uint4 v = q_s[32 * i];
                    qw[4 * i] = v.x; qw[4 * i + 1] = v.y; qw[4 * i + 2] = v.z; qw[4 * i + 3] = v.w;
                }
            }
#pragma unroll
            for (int gp = 0; gp < 2; ++gp) {                 // channels 32c + 16gp .. +15
                const uint4 ka = *reinterpret_cast<const uint4*>(kt + swz(g, 2 * c + gp));
                const uint4 kb = *reinterpret_cast<const uint4*>(kt + swz(g + 8, 2 * c + gp));
#pragma unroll
                for (int kk = 0; kk < 4; ++kk) {
                    const int ks = 4 * gp + kk;              // channels 32c + 4ks .. +3
                    const uint32_t wa = word_of(ka, kk), wb = word_of(kb, kk);
                    uint32_t A[4];
                    if constexpr (kInt8) {
                        const uint32_t xa = wa ^ 0x80808080u, xb = wb ^ 0x80808080u;
                        A[0] = s8x2_to_h2(xa, kSel01);
                        A[1] = s8x2_to_h2(xb, kSel01);
                        A[2] = s8x2_to_h2(xa, kSel23);
                        A[3] = s8x2_to_h2(xb, kSel23);
                    } else {
                        A[0] = e4m3x2_to_h2(wa);
                        A[1] = e4m3x2_to_h2(wb);
                        A[2] = e4m3x2_to_h2(wa >> 16);
                        A[3] = e4m3x2_to_h2(wb >> 16);
                    }
                    mma16816(dc, A, qw[2 * ks], qw[2 * ks + 1]);
                }
            }
            float sk[2] = {1.f, 1.f}, sv[2] = {1.f, 1.f};   // scales of tokens g, g+8
            if constexpr (kInt8) {
                float dd[4] = {0.f, 0.f, 0.f, 0.f};          // h' . q
#pragma unroll
                for (int gi = 0; gi < 4; ++gi) {             // a Philox call covers 8 channels
                    const uint4 da = philox((uint32_t)phys * kPage + g, c1, (uint32_t)(4 * c + gi), 0u, p.keys);
                    const uint4 db = philox((uint32_t)phys * kPage + g + 8, c1, (uint32_t)(4 * c + gi), 0u, p.keys);
#pragma unroll
                    for (int kk = 0; kk < 2; ++kk) {
                        const int ks = 2 * gi + kk;
                        const uint32_t H[4] = {h10(word_of(da, 2 * kk)), h10(word_of(db, 2 * kk)),
                                               h10(word_of(da, 2 * kk + 1)), h10(word_of(db, 2 * kk + 1))};
                        mma16816(dd, H, qw[2 * ks], qw[2 * ks + 1]);
                    }
                }
#pragma unroll
                for (int i = 0; i < 4; ++i) dc[i] = dc[i] - dd[i] + ((i & 1) ? zoff1 : zoff0);
                const __half* ks = reinterpret_cast<const __half*>(st + kOffKs);
                const __half* vs = reinterpret_cast<const __half*>(st + kOffVs);
                sk[0] = __half2float(ks[g]);
                sk[1] = __half2float(ks[g + 8]);
                sv[0] = __half2float(vs[g]);
                sv[1] = __half2float(vs[g + 8]);
            }

            // ---------------- logits, bound, softmax ------------------------------
            float cb[4] = {0.f, 0.f, 0.f, 0.f};
            {   // W . a_hi + W . a_lo in one product: W twice along k
                const uint32_t wa = *reinterpret_cast<const uint32_t*>(st + kOffW + (g * kBands + 2 * c) * 2);
                const uint32_t wb = *reinterpret_cast<const uint32_t*>(st + kOffW + ((g + 8) * kBands + 2 * c) * 2);
                const uint32_t A[4] = {wa, wb, wa, wb};
                mma16816(cb, A, a_hi, a_lo);
            }
            float y[4], P[4], cl[4];     // cl: the bounds in log2 units
            auto ub = [&](int i) { return ((i & 1) ? alpha1 : alpha0) * sk[i >> 1] * kLog2e; };   // Tier B's
#pragma unroll
            for (int i = 0; i < 4; ++i) {
                y[i] = kInt8 ? dc[i] * (sk[i >> 1] * kRsdLog2e) : dc[i] * kRsdLog2e;
                cl[i] = cb[i] * kLog2e;
            }
            // The value witness of tokens g, g+8 (0 past the context): fp8 loads it ahead of the
            // vote, the dithered cache, which has no registers to spare, behind it.
            float rho[2] = {0.f, 0.f}, vn[2] = {0.f, 0.f};
            auto load_vw = [&] {
                const float2 w0 = __half22float2(*reinterpret_cast<const __half2*>(st + kOffVw + 4 * g));
                const float2 w1 = __half22float2(*reinterpret_cast<const __half2*>(st + kOffVw + 4 * (g + 8)));
                rho[0] = w0.x;
                rho[1] = w1.x;
                vn[0] = w0.y;
                vn[1] = w1.y;
            };
            if constexpr (kValue && !kInt8) load_vw();
            // One warp vote finds everything that an ordinary page does not need: the
            // context's last page, a logit more than 8 above the reference, a V scale above the
            // P scale's limit, a bound of kHugeLog2 or more (meter_term).  Masks, six shuffles of
            // the maximum and the second vote on every page cost up to 2% (32 sequences of 1000
            // pages, 56 heads: 175.1 -> 172.9 us).
            auto largest = [&] {
                float m = fmaxf(fmaxf(cl[0], cl[1]), fmaxf(cl[2], cl[3]));
                if constexpr (kTierB) m = fmaxf(m, fmaxf(fmaxf(ub(0), ub(1)), fmaxf(ub(2), ub(3))));
                return m;
            };
            bool huge = false;
            if (__any_sync(0xffffffffu, nvalid < kPage || fmaxf(y[0], y[2]) > m_run[0] + 8.0f ||
                                            fmaxf(y[1], y[3]) > m_run[1] + 8.0f || !(largest() < kHugeLog2) ||
                                            (kInt8 && fmaxf(sv[0], sv[1]) >= sv_lim))) {
                const bool ok0 = g < nvalid, ok1 = g + 8 < nvalid;
#pragma unroll
                for (int i = 0; i < 4; ++i)
                    if (!((i >> 1) ? ok1 : ok0)) {   // tail slots may hold any bits
                        y[i] = -INFINITY;
                        cl[i] = 0.f;
                    }
                if (!ok0) sv[0] = sk[0] = rho[0] = vn[0] = 0.f;
                if (!ok1) sv[1] = sk[1] = rho[1] = vn[1] = 0.f;
                huge = __any_sync(0xffffffffu, largest() >= kHugeLog2);
                float mx0 = fmaxf(y[0], y[2]), mx1 = fmaxf(y[1], y[3]);
#pragma unroll
                for (int o = 4; o < 32; o <<= 1) {
                    mx0 = fmaxf(mx0, __shfl_xor_sync(0xffffffffu, mx0, o));
                    mx1 = fmaxf(mx1, __shfl_xor_sync(0xffffffffu, mx1, o));
                }
                const bool mv0 = mx0 > m_run[0] + 8.0f, mv1 = mx1 > m_run[1] + 8.0f;
                if (__any_sync(0xffffffffu, mv0 || mv1)) {
                    const float a0 = mv0 ? (m_run[0] == -INFINITY ? 0.f : fast_exp2(m_run[0] - mx0)) : 1.f;
                    const float a1 = mv1 ? (m_run[1] == -INFINITY ? 0.f : fast_exp2(m_run[1] - mx1)) : 1.f;
                    if (mv0) m_run[0] = mx0;
                    if (mv1) m_run[1] = mx1;
                    l_part[0] *= a0; d_part[0] *= a0;
                    l_part[1] *= a1; d_part[1] *= a1;
                    if constexpr (kTierB) { db_part[0] *= a0; db_part[1] *= a1; }
                    if constexpr (kInt8) { spv_part[0] *= a0; spv_part[1] *= a1; }
                    if constexpr (kValue) { vt_part[0] *= a0; vt_part[1] *= a1; }
#pragma unroll
                    for (int mt = 0; mt < 8; ++mt) {
                        acc[mt][0] *= a0; acc[mt][2] *= a0;
                        acc[mt][1] *= a1; acc[mt][3] *= a1;
                    }
                }
                if constexpr (kInt8) {
                    const float smax = fmaxf(sv[0], sv[1]);
                    if (__any_sync(0xffffffffu, smax >= sv_lim)) {
                        const float wmax = __int_as_float(__reduce_max_sync(0xffffffffu, __float_as_int(smax)));
                        const int want = 6 - (((__float_as_int(wmax) >> 23) & 0xFF) - 126);   // wmax < 2^(6 - want)
                        if (lam_exp != INT_MIN) {   // want < lam_exp here
                            const float f = pow2(want - lam_exp);
#pragma unroll
                            for (int mt = 0; mt < 8; ++mt)
#pragma unroll
                                for (int e2 = 0; e2 < 4; ++e2) acc[mt][e2] *= f;
                        }
                        lam_exp = want;
                        sv_lim = pow2(6 - lam_exp);
                    }
                }
            }
            if constexpr (kValue && kInt8) {
                load_vw();
                if (g >= nvalid) rho[0] = vn[0] = 0.f;
                if (g + 8 >= nvalid) rho[1] = vn[1] = 0.f;
            }
            if constexpr (kValue) vmax = fmaxf(vmax, fmaxf(vn[0], vn[1]));
            float dpg[2] = {0.f, 0.f};   // this page's share of D (kRepair)
#pragma unroll
            for (int i = 0; i < 4; ++i) {
                const int r = i >> 1, e = i & 1;
                const float pe = fast_exp2(y[i] - m_run[e]);     // 0 for masked tokens
                l_part[e] += pe;
                if (!huge) {
                    const float em1 = fast_exp2(cl[i]) - 1.f;
                    d_part[e] = fmaf(pe, em1, d_part[e]);
                    if constexpr (kRepair) dpg[e] = fmaf(pe, em1, dpg[e]);
                    if constexpr (kTierB) db_part[e] = fmaf(pe, fast_exp2(ub(i)) - 1.f, db_part[e]);
                }
                if constexpr (kValue) vt_part[e] = fmaf(pe, rho[r], vt_part[e]);
                P[i] = kInt8 ? pe * sv[r] : pe;
                if constexpr (kInt8) spv_part[e] += P[i];
            }
            if (huge) {
#pragma unroll
                for (int i = 0; i < 4; ++i) {
                    const int e = i & 1;
                    const float t = y[i] - m_run[e], dt = meter_term(t, cl[i]);
                    d_part[e] += dt;
                    if constexpr (kRepair) dpg[e] += dt;
                    if constexpr (kTierB) db_part[e] += meter_term(t, ub(i));
                }
            }
            if constexpr (kRepair) emit_page_terms(p, b, h, G, lp, g, c, dpg, m_run);
            // B = P^T for PV as two fp16 terms (hi + lo): the output is a sum with
            // heavy cancellation, one fp16 rounding of P is not accurate enough.
            // Packed as 8x8 blocks [token][head] (tokens 0-7 and 8-15) and
            // transposed with movmatrix into (P[tok 2c][head g], P[tok 2c+1][head g]).
            uint32_t bp0, bp1, bl0, bl1;
            {
                const float lam = pow2(kInt8 && lam_exp == INT_MIN ? 0 : lam_exp);
                const float x0 = P[0] * lam, x1 = P[1] * lam, x2 = P[2] * lam, x3 = P[3] * lam;
                const uint32_t h01 = pack_h2(x0, x1), h23 = pack_h2(x2, x3);
                const float2 r01 = __half22float2(*reinterpret_cast<const __half2*>(&h01));
                const float2 r23 = __half22float2(*reinterpret_cast<const __half2*>(&h23));
                const uint32_t l01 = pack_h2(x0 - r01.x, x1 - r01.y), l23 = pack_h2(x2 - r23.x, x3 - r23.y);
                bp0 = movmatrix_t(h01);
                bp1 = movmatrix_t(h23);
                bl0 = movmatrix_t(l01);
                bl1 = movmatrix_t(l23);
            }

            // ---------------- PV: acc[dim][head] ------------------------------------
            // The MMA truncates its sums: with the dither, whose terms nearly cancel, a page's are
            // taken from zero and added rounded (codes and dither apart: together they need
            // registers that are not there).
            auto add_pv = [&](int mt, const uint32_t (&A)[4]) {
                float page_sum[4] = {0.f, 0.f, 0.f, 0.f};
                float(&sum)[4] = kInt8 ? page_sum : acc[mt];
                mma16816(sum, A, bp0, bp1);
                mma16816(sum, A, bl0, bl1);
                if constexpr (kInt8) {
#pragma unroll
                    for (int i = 0; i < 4; ++i) acc[mt][i] += page_sum[i];
                }
            };
            const int tv[4] = {2 * c, 2 * c + 1, 2 * c + 8, 2 * c + 9};
            uint4 vq[4];
#pragma unroll
            for (int j = 0; j < 4; ++j) vq[j] = *reinterpret_cast<const uint4*>(kt + kTileRegion + swz(tv[j], g));
            if (!kInt8 && nvalid < kPage) {   // an fp8 NaN byte in an unused tail slot would poison P = 0 columns
#pragma unroll
                for (int j = 0; j < 4; ++j)
                    if (tv[j] >= nvalid) vq[j] = make_uint4(0, 0, 0, 0);
            }
#pragma unroll
            for (int mt = 0; mt < 8; ++mt) {
                const int wi = mt >> 1, pos = 2 * (mt & 1);
                uint32_t A[4];
#pragma unroll
                for (int pr = 0; pr < 2; ++pr) {
                    if constexpr (kInt8) {
                        const uint32_t X = prmt(word_of(vq[2 * pr], wi) ^ 0x80808080u,
                                                word_of(vq[2 * pr + 1], wi) ^ 0x80808080u, sel_interleave(pos));
                        A[2 * pr] = u8x2_minus(X, kSel01, kSubV);   // code + 1
                        A[2 * pr + 1] = u8x2_minus(X, kSel23, kSubV);
                    } else {
                        const uint32_t X = prmt(word_of(vq[2 * pr], wi), word_of(vq[2 * pr + 1], wi), sel_interleave(pos));
                        A[2 * pr] = e4m3x2_to_h2(X);
                        A[2 * pr + 1] = e4m3x2_to_h2(X >> 16);
                    }
                }
                add_pv(mt, A);
            }
            if constexpr (kInt8) {   // - H^T P^T
#pragma unroll
                for (int hf = 0; hf < 2; ++hf) {
                    uint4 dv[4];
#pragma unroll
                    for (int j = 0; j < 4; ++j)
                        dv[j] = philox((uint32_t)phys * kPage + tv[j], c1, (uint32_t)(2 * g + hf), 1u, p.keys);
#pragma unroll
                    for (int mm = 0; mm < 4; ++mm) {
                        uint32_t H[4];
#pragma unroll
                        for (int pr = 0; pr < 2; ++pr) {
                            const uint32_t wa = word_of(dv[2 * pr], mm), wb = word_of(dv[2 * pr + 1], mm);
                            H[2 * pr] = h10(prmt(wa, wb, 0x5410u)) | 0x80008000u;
                            H[2 * pr + 1] = h10(prmt(wa, wb, 0x7632u)) | 0x80008000u;
                        }
                        add_pv(4 * hf + mm, H);
                    }
                }
            }
        } else if constexpr (kRepair) {
            emit_skipped_page(p, b, h, G, lp, lane);
        }
        __syncwarp();
        issue(k + kStages, phys_issue);
        __syncwarp();
#pragma unroll
        for (int i = 0; i + 1 < kStages; ++i) ring[i] = ring[i + 1];
        ring[kStages - 1] = phys_issue;
    }
    if (failed) {
        // let copies still in flight land before the CTA's smem is released
        for (int k = consumed; k < min(n_my, consumed + kStages); ++k)
            (void)mbar_wait_bounded(&bars[k % kStages], (uint32_t)((k / kStages) & 1));
    }

    // ---- CTA merge: warps -> shared, one partial per CTA -----------------------------
    // a warp's totals for heads 2c, 2c+1 (reduced over the token rows g)
#pragma unroll
    for (int o = 4; o < 32; o <<= 1)
#pragma unroll
        for (int e = 0; e < 2; ++e) {
            l_part[e] += __shfl_xor_sync(0xffffffffu, l_part[e], o);
            d_part[e] += __shfl_xor_sync(0xffffffffu, d_part[e], o);
            if constexpr (kTierB) db_part[e] += __shfl_xor_sync(0xffffffffu, db_part[e], o);
            if constexpr (kInt8) spv_part[e] += __shfl_xor_sync(0xffffffffu, spv_part[e], o);
            if constexpr (kValue) vt_part[e] += __shfl_xor_sync(0xffffffffu, vt_part[e], o);
        }
    if constexpr (kValue)
        for (int o = 1; o < 32; o <<= 1) vmax = fmaxf(vmax, __shfl_xor_sync(0xffffffffu, vmax, o));
    __syncthreads();   // stage buffers are reused below
    float* mbuf = reinterpret_cast<float*>(smem);   // [warp][head][kPartialStride]
    {
        float* wb = mbuf + warp * kMaxGroup * kPartialStride;
        const float inv_lam = pow2(kInt8 && lam_exp == INT_MIN ? 0 : -lam_exp);
#pragma unroll
        for (int e = 0; e < 2; ++e) {
            float* row = wb + (2 * c + e) * kPartialStride + 16 * g;   // dims 16g .. 16g+15
            const float add = (kKappa - 1.0f) * spv_part[e];           // xi = h' - kappa, the codes raised by 1 (fp8: 0)
            auto out = [&](float x) { return kInt8 ? fmaf(x, inv_lam, add) : x * inv_lam; };
#pragma unroll
            for (int q4 = 0; q4 < 4; ++q4) {
                float4 v;
                v.x = out(acc[2 * q4][e]);
                v.y = out(acc[2 * q4][e + 2]);
                v.z = out(acc[2 * q4 + 1][e]);
                v.w = out(acc[2 * q4 + 1][e + 2]);
                *reinterpret_cast<float4*>(row + 4 * q4) = v;
            }
            if (g == 0) {
                wb[(2 * c + e) * kPartialStride + kHeadDim + 0] = m_run[e];
                wb[(2 * c + e) * kPartialStride + kHeadDim + 1] = l_part[e];
                wb[(2 * c + e) * kPartialStride + kHeadDim + 2] = d_part[e];
                if constexpr (kTierB) wb[(2 * c + e) * kPartialStride + kHeadDim + 3] = db_part[e];
                if constexpr (kValue) {
                    wb[(2 * c + e) * kPartialStride + kHeadDim + 4] = vt_part[e];
                    wb[(2 * c + e) * kPartialStride + kHeadDim + 5] = vmax;
                }
            }
        }
    }
    __syncthreads();
    const size_t unit = (size_t)b * p.num_kv_heads + h;
    float* part_out = p.partials + (unit * p.splits + split) * (kMaxGroup * kPartialStride);
    // thread -> (head, 4-dim chunk); chunk 32 carries (M, l, D)
    for (int idx = threadIdx.x; idx < G * 33; idx += kThreads) {
        const int hh = idx / 33, ch = idx % 33;
        float mw[kWarps];
        float M = -INFINITY;
#pragma unroll
        for (int w = 0; w < kWarps; ++w) {
            mw[w] = mbuf[(w * kMaxGroup + hh) * kPartialStride + kHeadDim];
            M = fmaxf(M, mw[w]);
        }
        float4 s = make_float4(0.f, 0.f, 0.f, 0.f);
        const int col = (ch < 32) ? 4 * ch : kHeadDim + 1;   // chunk 32: l, D
#pragma unroll
        for (int w = 0; w < kWarps; ++w) {
            if (mw[w] == -INFINITY) continue;   // a warp without pages: its values are not read
            const float wt = fast_exp2(mw[w] - M);
            const float* src = mbuf + (w * kMaxGroup + hh) * kPartialStride + col;
            if (ch < 32) {
                const float4 v = *reinterpret_cast<const float4*>(src);
                s.x = fmaf(wt, v.x, s.x); s.y = fmaf(wt, v.y, s.y);
                s.z = fmaf(wt, v.z, s.z); s.w = fmaf(wt, v.w, s.w);
            } else {
                s.x = fmaf(wt, src[0], s.x);   // l
                s.y = fmaf(wt, src[1], s.y);   // D
                if constexpr (kTierB) s.z = fmaf(wt, src[2], s.z);   // Tier-B D
                if constexpr (kValue) s.w = fmaf(wt, src[3], s.w);   // value term
            }
        }
        float* dst = part_out + hh * kPartialStride;
        if (ch < 32) {
            *reinterpret_cast<float4*>(dst + 4 * ch) = s;
        } else {
            dst[kHeadDim] = M;
            dst[kHeadDim + 1] = s.x;
            dst[kHeadDim + 2] = s.y;
            if constexpr (kTierB) dst[kHeadDim + 3] = s.z;
            if constexpr (kValue) {
                float vm = 0.f;
                for (int w = 0; w < kWarps; ++w)
                    vm = fmaxf(vm, mbuf[(w * kMaxGroup + hh) * kPartialStride + kHeadDim + 5]);
                dst[kHeadDim + 4] = s.w;
                dst[kHeadDim + 5] = vm;
            }
        }
    }
}

// ---------------------------------------------------------------------------
// Warp-specialized decode of the dithered INT8 cache.
//
// One CTA per SM with 8 consumer / 8 producer warp pairs.  Producer warp w
// serves consumer warp w through a 2-stage ring: it issues the page's copies
// (K and V code tiles by tensor-map TMA with the 128-byte swizzle, scales and
// witness by bulk copy) and regenerates the page's dither (Philox4x32-10) in
// registers, storing it as tiles j[token][channel] that the consumer reads with
// conflict-free 16-byte loads like the codes.  The consumer runs the attention,
// bound and meter math with no Philox on its path.  Per stage: `full` completes
// when the copies have landed and the dither tiles are written (two arrivals + the
// copy bytes); `empty` when the consumer has released it.  All waits are bounded.
//
// Measured (graph replay, us per call, before -> after in each case):
//  - the copies issued by an elected lane instead of lane 0 (their operands then stay
//    on the uniform path) together with K and V of a token drawn by the same lane, the
//    group constants of the first two Philox rounds kept, the bound as one MMA and one
//    vote a page for every rare case: 917 -> 875 warp instructions per page-head,
//    128k tokens x 4 heads 50.4 -> 48.2, 32k 17.06 -> 16.7;
//  - a warp index or page number that the compiler can prove uniform (a shuffle from
//    lane 0) undoes it: 1250 instructions per page-head and 66 us at 128k;
//  - the 10-bit dither here instead of in the consuming warps of the fp8 kernel's
//    layout: a batch of 4 x 1k-16k over 8 KV heads 82.5 -> 54.2.
// ---------------------------------------------------------------------------
constexpr int kWsPairs = 8;
// Built with -DWC_METER_OFF (a second library the benchmark loads to measure the
// certificate's cost, §8(d)): the warp-specialized decode then skips the
// witness copy, the bound MMAs and the meter accumulator; the meter it
// reports is not a bound.  The shipped library is built without it.
#ifdef WC_METER_OFF
constexpr bool kMeterOff = true;
#else
constexpr bool kMeterOff = false;
#endif
constexpr int kWsThreads = 64 * kWsPairs;
constexpr int kWsStages = 2;
// A stage: K codes | V codes [16][128] bytes (128-byte swizzle, 1024-aligned) | K
// dither | V dither | scales, witness, page header.  The dither tiles hold j: a
// byte a channel (8-bit dither, swizzled like the codes) or a 16-bit lane (10-bit,
// dither10_off).
template <int kBits>
struct WsStage {
    static constexpr int kDither = kBits == 8 ? 2048 : 4096;   // bytes of a dither tile
    static constexpr int kOffK = 0, kOffV = 2048, kOffKd = 4096, kOffVd = 4096 + kDither;
    static constexpr int kOffKs = 4096 + 2 * kDither;          // K scales [16] fp16
    static constexpr int kOffVs = kOffKs + 32;                 // V scales [16] fp16
    static constexpr int kOffW = kOffKs + 64;                  // witness [16][8] fp16
    static constexpr int kOffHdr = kOffKs + 320;               // physical page (or -1)
    static constexpr int kOffVw = kOffKs + 336;                // value witness [16][2] fp16 (value side)
    static constexpr int kBytes = kOffKs + 1024;
};
constexpr int kWsBarBytes = kWsPairs * kWsStages * 2 * 8;
// The CTA merge's buffer [warp][head][kPartialStride]: the stage area in the
// split plan, one of its own after the barriers in the flattened plan.  There
// the 10-bit stages (and the walkers' static slots) leave room for four heads at a
// time, their 128 outputs and six sums apart and without padding (two heads with
// it: 32 sequences of 8 to 60 pages, 8 x 8 heads, 40.0 -> 37.2 us).
template <int kBits, bool kFlat>
struct WsSmem {
    static constexpr int kStages = kWsPairs * kWsStages * WsStage<kBits>::kBytes;
    static constexpr bool kDense = kFlat && kBits == 10;
    static constexpr int kMergeHeads = kDense ? 4 : kMaxGroup;
    static constexpr int kMergeRow = kDense ? kHeadDim : kPartialStride;   // floats from row to row
    static constexpr int kMergeBytes = kWsPairs * kMergeHeads * (kDense ? kHeadDim + 6 : kPartialStride) * 4;
    static constexpr int kOffMerge = kFlat ? kStages + kWsBarBytes : 0;
    static constexpr int kBytes = kStages + kWsBarBytes + (kFlat ? kMergeBytes : 0) + 1024;   // + alignment slack
    static_assert(kBytes + (kFlat ? 1024 : 0) <= 232448, "shared memory limit of a CTA, static slots included");
    static_assert(kOffMerge % 16 == 0 && (kFlat || kMergeBytes <= kStages), "merge buffer");
};

// Byte offset of the 16-byte chunk q (8 channels) of token t in a 10-bit dither
// tile: two planes of 64 channels, [16 tokens][128 B] each.  The swizzle is
// injective over the token rows of each access: the producer's stores (4 tokens x 2
// halves a phase), the QK reads (2 tokens x 4 chunks in both planes) and ldmatrix
// (the 8 tokens of one k half).
__device__ __forceinline__ int dither10_off(int t, int q) {
    const int f = (t & 1) | (((t >> 1) ^ (t >> 2)) & 1) << 1 | ((t >> 3) & 1) << 2;
    return (q >> 3) * 2048 + t * 128 + (((q & 7) ^ f ^ ((q >> 3) << 1)) << 4);
}

struct WsParams {
    CUtensorMap k_map;   // k_codes as [num_pages * Hkv][16][128] bytes, box = one page of one head
    CUtensorMap v_map;
    DecodeParams p;
    WriteParams w;       // the cache as the write path sees it (append variant)
};

// Append (kXAppend): the step's new token of sequence b, the last of its
// context, is quantized and stored by the producer warp that stages the
// sequence's last page, before it issues the copies of the segment that holds
// that page.  Its slot must
// be that of the context's last token (else WC_DEV_BAD_APPEND, not written),
// so no other CTA reads it.  Lanes 0-7 hold the row (write path layout); the
// generic-proxy stores are fenced against the async-proxy copies that follow.
__device__ __forceinline__ void append_new_token(const WsParams& wp, int b, int h, int phys, int ctx, int lane) {
    const DecodeParams& p = wp.p;
    const int slot = load_dep(p.slot_new + b);
    if (slot < 0) return;   // warp-uniform: no new token for this sequence
    if (slot != phys * kPage + (ctx - 1) % kPage) {
        if (lane == 0) atomicOr(p.status, WC_DEV_BAD_APPEND);
        return;
    }
    const bool live = lane < 8;
    const int sub = lane & 7;
    const size_t off = ((size_t)b * p.num_kv_heads + h) * kHeadDim + sub * 16;
    uint4 rk[2] = {make_uint4(0, 0, 0, 0), make_uint4(0, 0, 0, 0)}, rv[2] = {rk[0], rk[1]};
    if (live) {
        rk[0] = load_dep(reinterpret_cast<const uint4*>(p.k_new + off));
        rk[1] = load_dep(reinterpret_cast<const uint4*>(p.k_new + off) + 1);
        rv[0] = load_dep(reinterpret_cast<const uint4*>(p.v_new + off));
        rv[1] = load_dep(reinterpret_cast<const uint4*>(p.v_new + off) + 1);
    }
    write_row<WC_SCHEME_DITHER_INT8, 8>(wp.w, rk, slot, live, h, 0, sub, nullptr, nullptr);
    write_row<WC_SCHEME_DITHER_INT8, 8>(wp.w, rv, slot, live, h, 1, sub, nullptr, nullptr);
    asm volatile("fence.proxy.async.global;" ::: "memory");
    __syncwarp();
}

__device__ __forceinline__ void consumer_sync() {   // the 8 consumer warps only
    asm volatile("bar.sync 1, %0;" ::"n"(32 * kWsPairs) : "memory");
}



template <int kBits, int kX>
__global__ void __launch_bounds__(kWsThreads, 1) decode_ws_kernel(const __grid_constant__ WsParams wp) {
    constexpr bool kTierB = (kX & kXTierB) != 0, kValue = (kX & kXValue) != 0, kRepair = (kX & kXRepair) != 0;
    constexpr bool kAppend = (kX & kXAppend) != 0;
    constexpr bool kFlat = (kX & kXFlat) != 0;   // flattened split plan (pages_per_split == 0)
    constexpr bool kStall = (kX & kXStall) != 0;
    constexpr int kTries = kStall ? kStallTries : kMaxWaitTries;
    const DecodeParams& p = wp.p;
    extern __shared__ __align__(1024) uint8_t smem_raw[];
    uint8_t* smem = smem_raw + ((1024 - (smem_addr(smem_raw) & 1023)) & 1023);
    const int lane = threadIdx.x & 31, warp = threadIdx.x >> 5;
    const bool producer = warp >= kWsPairs;
    const int pw = producer ? warp - kWsPairs : warp;     // pair index
    const int g = lane >> 2, c = lane & 3;
    const int G = p.group;
    using St = WsStage<kBits>;
    using Sm = WsSmem<kBits, kFlat>;
    constexpr float kKappaK = DitherConst<kBits>::kappa;
    // V codes enter the MMAs raised by beta, the whole part of h' (4, or 1 with the
    // 10-bit dither), so the PV sums carry a bias below 1/2 a token
    constexpr float kKappaV = DitherConst<kBits>::kappa - (kBits == 8 ? 4.0f : 1.0f);
    constexpr uint32_t kSubV = kBits == 8 ? 0x647C647Cu : 0x647F647Fu;   // 1152 - beta

    uint8_t* stages = smem + pw * kWsStages * St::kBytes;
    uint64_t* full = reinterpret_cast<uint64_t*>(smem + Sm::kStages) + pw * 2 * kWsStages;
    uint64_t* empty = full + kWsStages;
    if (kBits == 10 && threadIdx.x == 32 * kWsPairs) {   // 10-bit: 1.6% off a step; 8-bit: nothing
        prefetch_map(&wp.k_map);
        prefetch_map(&wp.v_map);
    }
    if (producer && lane == 0)
        for (int s = 0; s < kWsStages; ++s) {
            mbar_init(&full[s], 2);
            mbar_init(&empty[s], 1);
        }
    fence_barrier_init();
    __syncthreads();   // every barrier is initialised before any warp waits on it
    // the dependent merge may be scheduled now: it waits for this whole grid
    // (griddepcontrol.wait), and it launches only once every CTA of this grid
    // has started, so its CTAs never hold resources this grid still needs
    grid_dep_launch();
    if (!kFlat && lane == 0 && p.max_pages > 0) {
        // Split plan.  While the preceding kernel drains: warm L2 with this pair's
        // first page and the CTA's query rows.  The context length and page-table
        // entry read here may still be changing, so they serve only as prefetch
        // addresses (clamped into the cache); the loads bypass L1, which therefore
        // holds no copy that the reads after the wait could hit.
        const int b = blockIdx.z, h = blockIdx.y, p0 = blockIdx.x * p.pages_per_split;
        if (producer) {
            const int ctx_hint = __ldcg(p.ctx_lens + b);
            if (p0 + pw < p.max_pages && (p0 + pw) * kPage < ctx_hint) warm_page(p, b, h, p0 + pw, 32);
        } else if (pw == 0) {
            warm_queries(p, b, h);
        }
    }
    // q, page tables and the cache may come from the preceding kernel (the flattened plan waits below)
    if constexpr (!kFlat) grid_dep_wait();

    // Split plan: this pair's first page-table entry and the consumer's query
    // fragment are loaded alongside the context length (both in bounds
    // whatever the length; used only if the pair has pages).
    int phys_first = -1;
    uint32_t qw[16];
    if constexpr (!kFlat) {
        if (producer && p.max_pages > 0)
            phys_first = load_dep(p.block_table + (size_t)blockIdx.z * p.max_pages +
                               min((int)blockIdx.x * p.pages_per_split + pw, p.max_pages - 1));
        if (!producer) load_q_frag(p, blockIdx.z, blockIdx.y, G, g, c, qw);
    }
    WsSeg sg;
    bool have;
    WsSeg* my_seg = nullptr;   // flattened plan: this warp's walker, in shared memory
    if constexpr (kFlat) {
        __shared__ FlatScratch s_flat;
        __shared__ WsSeg s_seg[kWsThreads / 32];
        have = flat_plan(p, sg, s_flat, [&](const WsSeg& hint) {
            if (lane != 0) return;
            if (producer) {
                if (hint.a + pw < hint.e) warm_page(p, hint.b, hint.h, hint.a + pw, 32);
            } else if (pw == 0) {
                warm_queries(p, hint.b, hint.h);
            }
        });
        my_seg = &s_seg[warp];
        if (lane == 0) *my_seg = sg;
        __syncwarp();
    } else {
        split_segment(p, sg);
        have = true;
    }

    if (producer) {
        int k = 0, issued = 0;   // stage ring position, continued across segments
        bool stop = false;
        const int pt = lane >> 1, hf = lane & 1;
        PhiloxGroup grp[kBits == 8 ? 1 : 2][4];   // a CTA's segments share their KV head
        {
            const int hk = kFlat ? (int)blockIdx.x % p.num_kv_heads : (int)blockIdx.y;
            const uint32_t c1 = (uint32_t)p.layer * 65536u + (uint32_t)hk;
#pragma unroll
            for (int j = 0; j < 4; ++j) {
                if constexpr (kBits == 8) {
                    grp[0][j] = philox_group((uint32_t)(4 * hf + j), c1, p.keys);
                } else {
                    grp[0][j] = philox_group((uint32_t)(8 * hf + 4 * hf + j), c1, p.keys);
                    grp[1][j] = philox_group((uint32_t)(8 * hf + 4 * (hf ^ 1) + j), c1, p.keys);
                }
            }
        }
        // one segment's pages (the split plan has one segment: no loop around it)
        auto produce = [&](const WsSeg& cs) {
            const int b = cs.b, h = cs.h, ctx = cs.ctx, npages = cs.np;
            const int32_t* bt_row = p.block_table + (size_t)b * p.max_pages;
            int first;
            const int n_seg = ws_seg_pages<kWsPairs>(cs, pw, first);
            int phys_next = kFlat ? (n_seg > 0 ? load_dep(bt_row + first) : -1) : phys_first;
            if constexpr (kAppend) {
                // The stream that stages the sequence's last page in this segment stores
                // the new token before the segment's first page (not inside the page
                // loop), so its write overlaps the other streams' pages and the loop
                // carries no write code.  Its copies are issued after the token's stores.
                const int lpl = npages - 1;
                if (n_seg > 0 && lpl >= first && (lpl - first) % kWsPairs == 0 && lpl < cs.e) {
                    const int phl = load_dep(bt_row + lpl);
                    if (phl >= 0 && phl < p.num_pages) append_new_token(wp, b, h, phl, ctx, lane);
                }
            }
            for (int i = 0; i < n_seg; ++i, ++k) {
                const int lp = first + kWsPairs * i;
                const int s = k % kWsStages;
                if (k >= kWsStages) {
                    const bool freed = mbar_wait_bounded<kTries>(&empty[s], (uint32_t)(((k / kWsStages) - 1) & 1));
                    if (!__all_sync(0xffffffffu, freed)) {
                        if (lane == 0) atomicOr(p.status, WC_DEV_TIMEOUT);
                        stop = true;
                        break;
                    }
                }
                const int phys = phys_next;
                if (i + 1 < n_seg) phys_next = load_dep(bt_row + lp + kWsPairs);
                const bool ok = phys >= 0 && phys < p.num_pages;
                uint8_t* st = stages + s * St::kBytes;
                if constexpr (kStall) {   // failure-detection test: this page is never staged
                    if (lp == p.stall_page) {
                        issued = k + 1;
                        continue;
                    }
                }
                // one elected lane (not a lane test): the copies' operands then stay on
                // the uniform path
                if (elect_one()) {
                    *reinterpret_cast<int*>(st + St::kOffHdr) = ok ? phys : -1;
                    if (ok) {
                        const int z = phys * p.num_kv_heads + h;
                        const size_t ph = (size_t)z;
                        mbar_arrive_expect_tx(&full[s],
                                              (uint32_t)(kStageBytes - (kMeterOff ? 256 : 0) + (kValue ? 64 : 0)));
                        tma_page(st + St::kOffK, &wp.k_map, z, &full[s]);
                        tma_page(st + St::kOffV, &wp.v_map, z, &full[s]);
                        bulk_g2s(st + St::kOffKs, p.k_scale + ph * kPage, 32, &full[s]);
                        bulk_g2s(st + St::kOffVs, p.v_scale + ph * kPage, 32, &full[s]);
                        if constexpr (!kMeterOff)
                            bulk_g2s(st + St::kOffW, p.k_witness + ph * (kPage * kBands), 256, &full[s]);
                        if constexpr (kValue) bulk_g2s(st + St::kOffVw, p.v_witness + ph * (kPage * 2), 64, &full[s]);
                    } else {
                        atomicOr(p.status, WC_DEV_BAD_PAGE);
                        asm volatile("mbarrier.arrive.shared::cta.b64 _, [%0];" ::"r"(smem_addr(&full[s])) : "memory");
                    }
                }
                issued = k + 1;
                if (ok) {
                    // Dither of K and V of one token per lane pair: lane 2t + hf draws token t's
                    // channels 64 hf .. +63 (four counter groups at a time, K and V together).
                    const uint32_t slot = (uint32_t)phys * kPage + pt;
                    if constexpr (kBits == 8) {
                        uint32_t w[2][4][4];
                        philox_kv(slot, grp[0], p.keys, w);
#pragma unroll
                        for (int j = 0; j < 4; ++j) {
                            const int off = swz(pt, 4 * hf + j);
                            *reinterpret_cast<uint4*>(st + St::kOffKd + off) =
                                make_uint4(w[0][j][0], w[0][j][1], w[0][j][2], w[0][j][3]);
                            *reinterpret_cast<uint4*>(st + St::kOffVd + off) =
                                make_uint4(w[1][j][0], w[1][j][1], w[1][j][2], w[1][j][3]);
                        }
                    } else {
#pragma unroll
                        for (int bt = 0; bt < 2; ++bt) {
                            uint32_t w[2][4][4];
                            philox_kv(slot, grp[bt], p.keys, w);
#pragma unroll
                            for (int j = 0; j < 4; ++j) {
                                const int off = dither10_off(pt, 8 * hf + 4 * (bt ^ hf) + j);
                                *reinterpret_cast<uint4*>(st + St::kOffKd + off) =
                                    make_uint4(w[0][j][0], w[0][j][1], w[0][j][2], w[0][j][3]);
                                *reinterpret_cast<uint4*>(st + St::kOffVd + off) =
                                    make_uint4(w[1][j][0], w[1][j][1], w[1][j][2], w[1][j][3]);
                            }
                        }
                    }
                }
                __syncwarp();
                if (lane == 0)   // second arrival: dither tiles and header are written
                    asm volatile("mbarrier.arrive.shared::cta.b64 _, [%0];" ::"r"(smem_addr(&full[s])) : "memory");
            }
        };
        if constexpr (kFlat) {
            for (bool more = have; more && !stop; more = ws_step<kWsPairs>(p, my_seg, lane)) produce(*my_seg);
        } else {
            produce(sg);
        }
        // copies still in flight must land before the CTA's smem is released
        for (int j = max(0, issued - kWsStages); j < issued; ++j)
            (void)mbar_wait_bounded<kTries>(&full[j % kWsStages], (uint32_t)((j / kWsStages) & 1));
        return;
    }

    // ---------------------------- consumer warps ------------------------------------
    // The CTA merge's buffer [warp][head][kPartialStride]: the stage area in the
    // split plan (one segment, the producers are done with it), a buffer of its
    // own in the flattened plan (the producers stage the next segment meanwhile).
    float* mbuf = reinterpret_cast<float*>(smem + Sm::kOffMerge);
    // Token rows: row g of the QK and softmax tiles holds token t0, row g + 8
    // token t1 (tok_row), so that the P fragment transposed by movmatrix pairs
    // tokens (4c, 4c+1) and (4c+2, 4c+3), as ldmatrix.trans delivers V.
    const int t0 = tok_row(g), t1 = tok_row(g + 8);
    int k = 0;   // stage ring position, continued across segments
    bool failed = false;
    // one segment: query setup, pages, CTA merge (the split plan has one segment)
    auto consume = [&](const WsSeg& cs) {
        const int b = cs.b, h = cs.h, ctx = cs.ctx;
        const bool row_valid = g < G;
        if constexpr (kFlat) {
            load_q_frag(p, b, h, G, g, c, qw);
            if (pw == 0 && lane == 0 && cs.vb + cs.np + kCutPages < cs.hi && b + 1 < p.batch)
                warm_queries(p, b + 1, h);   // of the next segment (or of a sequence without pages)
        }
        float qsum = 0.f, part[4] = {0.f, 0.f, 0.f, 0.f};
#pragma unroll
        for (int i = 0; i < 16; ++i) {
            const float2 f = __half22float2(*reinterpret_cast<const __half2*>(&qw[i]));
            qsum += f.x + f.y;
            part[i >> 2] = fmaf(f.x, f.x, fmaf(f.y, f.y, part[i >> 2]));
        }
        qsum += __shfl_xor_sync(0xffffffffu, qsum, 1);
        qsum += __shfl_xor_sync(0xffffffffu, qsum, 2);
        // Tier B (§4.2): u_t = alpha s_t with alpha = sqrt(2 log(2S/delta) ||q||^2 / (12 d)),
        // for this thread's softmax heads 2c and 2c+1
        float alpha0 = 0.f, alpha1 = 0.f;
        if constexpr (kTierB) {
            float qn2 = part[0] + part[1] + part[2] + part[3];   // ||q_g||^2 over channels 32c .. 32c+31
            qn2 += __shfl_xor_sync(0xffffffffu, qn2, 1);
            qn2 += __shfl_xor_sync(0xffffffffu, qn2, 2);
            const float lg = p.tb_log_2_over_delta + logf((float)max(ctx, 1));   // log(2S / delta)
            const float al = sqrtf(2.0f * lg * qn2 * (1.0f / (12.0f * kHeadDim)));
            alpha0 = __shfl_sync(0xffffffffu, al, 8 * c);
            alpha1 = __shfl_sync(0xffffffffu, al, 8 * c + 4);
        }
        float band_a, band_b;
        if (p.rope_layout == WC_ROPE_HALF) {
#pragma unroll
            for (int i = 0; i < 4; ++i) part[i] += __shfl_xor_sync(0xffffffffu, part[i], 2);
            const int src = (lane & ~3) | (c >> 1);
            float v[4];
#pragma unroll
            for (int i = 0; i < 4; ++i) v[i] = __shfl_sync(0xffffffffu, part[i], src);
            band_a = (c & 1) ? v[2] : v[0];
            band_b = (c & 1) ? v[3] : v[1];
        } else {
            band_a = part[0] + part[1];
            band_b = part[2] + part[3];
        }
        uint32_t a_hi = 0, a_lo = 0;   // ||q_b|| log2(e) / sqrt(d), hi + lo: the bound in log2 units
        if (row_valid) {
            const float x0 = sqrtf(band_a) * kRsdLog2e, x1 = sqrtf(band_b) * kRsdLog2e;
            const __half h0 = __float2half_rn(x0), h1 = __float2half_rn(x1);
            a_hi = pack_h2(__half2float(h0), __half2float(h1));
            a_lo = pack_h2(x0 - __half2float(h0), x1 - __half2float(h1));
        }
        const float zoff0 = kKappaK * __shfl_sync(0xffffffffu, qsum, 8 * c);
        const float zoff1 = kKappaK * __shfl_sync(0xffffffffu, qsum, 8 * c + 4);

        float m_run[2] = {-INFINITY, -INFINITY};
        float l_part[2] = {0.f, 0.f}, d_part[2] = {0.f, 0.f}, spv_part[2] = {0.f, 0.f};
        float db_part[2] = {0.f, 0.f};   // Tier-B meter accumulator (kTierB)
        float vt_part[2] = {0.f, 0.f};   // value side: sum p~ rho^v (kValue)
        float vmax = 0.f;                // value side: max ||v|| over this thread's tokens
        float acc[8][4];
#pragma unroll
        for (int i = 0; i < 8; ++i) acc[i][0] = acc[i][1] = acc[i][2] = acc[i][3] = 0.f;
        // P * s_v * 2^lam_exp stays below 2^14 (fp16): s_v * 2^lam_exp < 2^6.  lam_exp only
        // decreases; sv_lim = 2^(6 - lam_exp) is the scale at which it must, FLT_MIN
        // until the first positive scale.
        int lam_exp = INT_MIN;
        float lam = 1.f, sv_lim = 1.17549435e-38f;

        int first;
        const int n_seg = ws_seg_pages<kWsPairs>(cs, pw, first);
        for (int i = 0; i < n_seg && !failed; ++i, ++k) {
            const int s = k % kWsStages;
            const bool landed = mbar_wait_bounded<kTries>(&full[s], (uint32_t)((k / kWsStages) & 1));
            if (!__all_sync(0xffffffffu, landed)) {
                if (lane == 0) atomicOr(p.status, WC_DEV_TIMEOUT);
                failed = true;   // later pages are not waited for; the merges still run
                break;
            }
            const uint8_t* st = stages + s * St::kBytes;
            const int lp = first + kWsPairs * i;

            // ---------------- QK: S[token][head] = code.q - h'.q -------------------
            // Row g of the QK tile holds token t0, row g + 8 token t1 (see tok_row).  (A page
            // outside the pool leaves any bits here; it is skipped below.)
            float dc[4] = {0.f, 0.f, 0.f, 0.f}, dd[4] = {0.f, 0.f, 0.f, 0.f};
#pragma unroll
            for (int gp = 0; gp < 2; ++gp) {
                const int q16 = 2 * c + gp;   // 16-byte chunk: channels 32c + 16gp .. +15
                const uint4 ka = *reinterpret_cast<const uint4*>(st + St::kOffK + swz(t0, q16));
                const uint4 kb = *reinterpret_cast<const uint4*>(st + St::kOffK + swz(t1, q16));
                uint4 ja[kBits == 8 ? 1 : 2], jb[kBits == 8 ? 1 : 2];
                if constexpr (kBits == 8) {
                    ja[0] = *reinterpret_cast<const uint4*>(st + St::kOffKd + swz(t0, q16));
                    jb[0] = *reinterpret_cast<const uint4*>(st + St::kOffKd + swz(t1, q16));
                } else {
#pragma unroll
                    for (int x = 0; x < 2; ++x) {
                        ja[x] = *reinterpret_cast<const uint4*>(st + St::kOffKd + dither10_off(t0, 2 * q16 + x));
                        jb[x] = *reinterpret_cast<const uint4*>(st + St::kOffKd + dither10_off(t1, 2 * q16 + x));
                    }
                }
#pragma unroll
                for (int kk = 0; kk < 4; ++kk) {
                    const int ks = 4 * gp + kk;
                    const uint32_t xa = word_of(ka, kk) ^ 0x80808080u, xb = word_of(kb, kk) ^ 0x80808080u;
                    const uint32_t A[4] = {s8x2_to_h2(xa, kSel01), s8x2_to_h2(xb, kSel01), s8x2_to_h2(xa, kSel23),
                                           s8x2_to_h2(xb, kSel23)};
                    mma16816(dc, A, qw[2 * ks], qw[2 * ks + 1]);
                    if constexpr (kBits == 8) {
                        const uint32_t ya = word_of(ja[0], kk), yb = word_of(jb[0], kk);
                        const uint32_t H[4] = {h8(ya, kSel01), h8(yb, kSel01), h8(ya, kSel23), h8(yb, kSel23)};
                        mma16816(dd, H, qw[2 * ks], qw[2 * ks + 1]);
                    } else {
                        const uint4 &va = ja[kk >> 1], &vb = jb[kk >> 1];
                        const int x = 2 * (kk & 1);
                        const uint32_t H[4] = {h10(word_of(va, x)), h10(word_of(vb, x)), h10(word_of(va, x + 1)),
                                               h10(word_of(vb, x + 1))};
                        mma16816(dd, H, qw[2 * ks], qw[2 * ks + 1]);
                    }
                }
            }

            // ---------------- logits, bound, softmax ------------------------------
            float cb[4] = {0.f, 0.f, 0.f, 0.f};   // log2-domain bound (a carries log2 e)
            if constexpr (!kMeterOff) {   // W . a_hi + W . a_lo in one product: W twice along k
                const uint32_t wa = *reinterpret_cast<const uint32_t*>(st + St::kOffW + (t0 * kBands + 2 * c) * 2);
                const uint32_t wb = *reinterpret_cast<const uint32_t*>(st + St::kOffW + (t1 * kBands + 2 * c) * 2);
                const uint32_t A[4] = {wa, wb, wa, wb};
                mma16816(cb, A, a_hi, a_lo);
            }
            const __half* ksc = reinterpret_cast<const __half*>(st + St::kOffKs);
            const __half* vsc = reinterpret_cast<const __half*>(st + St::kOffVs);
            float sk[2] = {__half2float(ksc[t0]), __half2float(ksc[t1])};
            float sv[2] = {__half2float(vsc[t0]), __half2float(vsc[t1])};
            float y[4];
#pragma unroll
            for (int i2 = 0; i2 < 4; ++i2) {
                const int r = i2 >> 1, e = i2 & 1;
                y[i2] = (dc[i2] - dd[i2] + (e ? zoff1 : zoff0)) * (sk[r] * kRsdLog2e);
            }
            float rho[2] = {0.f, 0.f};   // value witness of tokens t0, t1 (0 past the context)
            float vn[2] = {0.f, 0.f};
            if constexpr (kValue) {
                const float2 w0 = __half22float2(*reinterpret_cast<const __half2*>(st + St::kOffVw + 4 * t0));
                const float2 w1 = __half22float2(*reinterpret_cast<const __half2*>(st + St::kOffVw + 4 * t1));
                rho[0] = w0.x;
                rho[1] = w1.x;
                vn[0] = w0.y;
                vn[1] = w1.y;
            }
            float ub[4];                 // Tier-B bound in log2 units (kTierB)
#pragma unroll
            for (int i2 = 0; i2 < 4; ++i2) ub[i2] = kTierB ? ((i2 & 1) ? alpha1 : alpha0) * sk[i2 >> 1] * kLog2e : 0.f;
            float big = kMeterOff ? 0.f : fmaxf(fmaxf(cb[0], cb[1]), fmaxf(cb[2], cb[3]));
            if constexpr (kTierB) big = fmaxf(big, fmaxf(fmaxf(ub[0], ub[1]), fmaxf(ub[2], ub[3])));
            // One warp vote finds everything that an ordinary page does not need: a page
            // outside the pool, the context's last page, a logit more than 8 above the
            // reference, a V scale above the P scale's limit, a bound of kHugeLog2 or more.
            const int page = *reinterpret_cast<const int*>(st + St::kOffHdr);
            bool skip = false, huge = false;
            if (__any_sync(0xffffffffu, page < 0 || (lp + 1) * kPage > ctx || fmaxf(y[0], y[2]) > m_run[0] + 8.0f ||
                                            fmaxf(y[1], y[3]) > m_run[1] + 8.0f || fmaxf(sv[0], sv[1]) >= sv_lim ||
                                            !(big < kHugeLog2))) {
                skip = page < 0;
                const int nvalid = min(kPage, ctx - lp * kPage);
                if (!skip) {
                    if (nvalid < kPage) {   // slots past the context hold any bits
                        const bool ok0 = t0 < nvalid, ok1 = t1 < nvalid;
#pragma unroll
                        for (int i2 = 0; i2 < 4; ++i2)
                            if (!((i2 >> 1) ? ok1 : ok0)) {
                                y[i2] = -INFINITY;
                                cb[i2] = ub[i2] = 0.f;
                            }
                        if (!ok0) sv[0] = sk[0] = rho[0] = vn[0] = 0.f;
                        if (!ok1) sv[1] = sk[1] = rho[1] = vn[1] = 0.f;
                        big = fmaxf(fmaxf(cb[0], cb[1]), fmaxf(cb[2], cb[3]));
                        if constexpr (kTierB) big = fmaxf(big, fmaxf(fmaxf(ub[0], ub[1]), fmaxf(ub[2], ub[3])));
                    }
                    huge = __any_sync(0xffffffffu, big >= kHugeLog2);
                    // running maximum, moved lazily: only when a logit exceeds it by more than 8
                    float mx0 = fmaxf(y[0], y[2]), mx1 = fmaxf(y[1], y[3]);
                    if (__any_sync(0xffffffffu, mx0 > m_run[0] + 8.0f || mx1 > m_run[1] + 8.0f)) {
#pragma unroll
                        for (int o = 4; o < 32; o <<= 1) {
                            mx0 = fmaxf(mx0, __shfl_xor_sync(0xffffffffu, mx0, o));
                            mx1 = fmaxf(mx1, __shfl_xor_sync(0xffffffffu, mx1, o));
                        }
                        const bool mv0 = mx0 > m_run[0] + 8.0f, mv1 = mx1 > m_run[1] + 8.0f;
                        const float a0 = mv0 ? (m_run[0] == -INFINITY ? 0.f : fast_exp2(m_run[0] - mx0)) : 1.f;
                        const float a1 = mv1 ? (m_run[1] == -INFINITY ? 0.f : fast_exp2(m_run[1] - mx1)) : 1.f;
                        if (mv0) m_run[0] = mx0;
                        if (mv1) m_run[1] = mx1;
                        l_part[0] *= a0; d_part[0] *= a0; spv_part[0] *= a0;
                        l_part[1] *= a1; d_part[1] *= a1; spv_part[1] *= a1;
                        if constexpr (kTierB) { db_part[0] *= a0; db_part[1] *= a1; }
                        if constexpr (kValue) { vt_part[0] *= a0; vt_part[1] *= a1; }
#pragma unroll
                        for (int mt = 0; mt < 8; ++mt) {
                            acc[mt][0] *= a0; acc[mt][2] *= a0;
                            acc[mt][1] *= a1; acc[mt][3] *= a1;
                        }
                    }
                    if (__any_sync(0xffffffffu, fmaxf(sv[0], sv[1]) >= sv_lim)) {
                        const float smax = fmaxf(sv[0], sv[1]);
                        const float wmax = __int_as_float(__reduce_max_sync(0xffffffffu, __float_as_int(smax)));
                        const int e = ((__float_as_int(wmax) >> 23) & 0xFF) - 126;   // wmax < 2^e
                        const int want = 6 - e;
                        if (lam_exp != INT_MIN) {   // want < lam_exp here
                            const float f = pow2(want - lam_exp);
#pragma unroll
                            for (int mt = 0; mt < 8; ++mt)
#pragma unroll
                                for (int e2 = 0; e2 < 4; ++e2) acc[mt][e2] *= f;
                            spv_part[0] *= f;
                            spv_part[1] *= f;
                        }
                        lam_exp = want;
                        lam = pow2(lam_exp);
                        sv_lim = pow2(6 - lam_exp);
                    }
                } else if constexpr (kRepair) {
                    emit_skipped_page(p, b, h, G, lp, lane);
                }
            }
            if (!skip) {
                const float svl[2] = {sv[0] * lam, sv[1] * lam};   // exact: lam is a power of two
                if constexpr (kValue) vmax = fmaxf(vmax, fmaxf(vn[0], vn[1]));
                float dpg[2] = {0.f, 0.f};   // this page's share of D (kRepair)
                float x[4];                  // P * s_v * lam, the PV operand
#pragma unroll
                for (int i2 = 0; i2 < 4; ++i2) {
                    const int r = i2 >> 1, e = i2 & 1;
                    const float pe = fast_exp2(y[i2] - m_run[e]);
                    l_part[e] += pe;
                    if (!huge) {
                        if constexpr (!kMeterOff) {
                            const float em1 = fast_exp2(cb[i2]) - 1.f;
                            d_part[e] = fmaf(pe, em1, d_part[e]);
                            if constexpr (kRepair) dpg[e] = fmaf(pe, em1, dpg[e]);
                        }
                        if constexpr (kTierB) db_part[e] = fmaf(pe, fast_exp2(ub[i2]) - 1.f, db_part[e]);
                    }
                    if constexpr (kValue) vt_part[e] = fmaf(pe, rho[r], vt_part[e]);
                    x[i2] = pe * svl[r];
                    spv_part[e] += x[i2];     // sum P s_v, in the lam frame
                }
                if (huge) {
#pragma unroll
                    for (int i2 = 0; i2 < 4; ++i2) {
                        const int e = i2 & 1;
                        const float t = y[i2] - m_run[e];
                        if constexpr (!kMeterOff) {
                            const float dt = meter_term(t, cb[i2]);
                            d_part[e] += dt;
                            if constexpr (kRepair) dpg[e] += dt;
                        }
                        if constexpr (kTierB) db_part[e] += meter_term(t, ub[i2]);
                    }
                }
                if constexpr (kRepair) emit_page_terms(p, b, h, G, lp, g, c, dpg, m_run);
                uint32_t bp0, bp1, bl0, bl1;
                {
                    const uint32_t h01 = pack_h2(x[0], x[1]), h23 = pack_h2(x[2], x[3]);
                    const float2 r01 = __half22float2(*reinterpret_cast<const __half2*>(&h01));
                    const float2 r23 = __half22float2(*reinterpret_cast<const __half2*>(&h23));
                    const uint32_t l01 = pack_h2(x[0] - r01.x, x[1] - r01.y), l23 = pack_h2(x[2] - r23.x, x[3] - r23.y);
                    // B operand: P[tokens 4c, 4c+1][head g] and P[tokens 4c+2, 4c+3][head g]
                    bp0 = movmatrix_t(h01);
                    bp1 = movmatrix_t(h23);
                    bl0 = movmatrix_t(l01);
                    bl1 = movmatrix_t(l23);
                }

                // ---------------- PV: acc[dim][head] += (code + beta - h') P -----------
                // ldmatrix.trans of a 16x16 byte block (tokens x dims 16mt..16mt+15)
                // gives lane (g, c) dims 16mt + g (first word) and 16mt + g + 8 (second)
                // at tokens 4c .. 4c+3: the A operand with k slots 2c, 2c+1, 2c+8,
                // 2c+9 holding tokens 4c .. 4c+3, the order B was built in.  The 10-bit
                // dither's 16-bit lanes come by the b16 form from the same token rows.
#pragma unroll
                for (int mp = 0; mp < 4; ++mp) {   // m-tiles 2mp, 2mp+1
                    uint32_t v[4], j[4];
                    ldsm_t_b8_x2(v, st + St::kOffV + swz(lane & 15, 2 * mp + (lane >> 4)));
                    if constexpr (kBits == 8) ldsm_t_b8_x2(j, st + St::kOffVd + swz(lane & 15, 2 * mp + (lane >> 4)));
#pragma unroll
                    for (int u = 0; u < 2; ++u) {
                        const int mt = 2 * mp + u;
                        const uint32_t x0 = v[2 * u] ^ 0x80808080u, x1 = v[2 * u + 1] ^ 0x80808080u;
                        const uint32_t A[4] = {u8x2_minus(x0, kSel01, kSubV), u8x2_minus(x1, kSel01, kSubV),
                                               u8x2_minus(x0, kSel23, kSubV), u8x2_minus(x1, kSel23, kSubV)};
                        // The MMA truncates its sums.  With the 10-bit dither a page is summed on
                        // its own and added rounded: that kernel's streams took half as many pages
                        // each before they were paired with a producer.
                        float page_sum[4] = {0.f, 0.f, 0.f, 0.f};
                        float(&sum)[4] = kBits == 8 ? acc[mt] : page_sum;
                        mma16816(sum, A, bp0, bp1);
                        mma16816(sum, A, bl0, bl1);
                        uint32_t H[4];
                        if constexpr (kBits == 8) {
                            H[0] = nh8(j[2 * u], kSel01);
                            H[1] = nh8(j[2 * u + 1], kSel01);
                            H[2] = nh8(j[2 * u], kSel23);
                            H[3] = nh8(j[2 * u + 1], kSel23);
                        } else {
                            ldsm_t_b16_x4(H, st + St::kOffVd + dither10_off(tok_row((lane & 7) + 8 * (lane >> 4)),
                                                                            2 * mt + ((lane >> 3) & 1)));
#pragma unroll
                            for (int x2 = 0; x2 < 4; ++x2) H[x2] = h10(H[x2]) | 0x80008000u;
                        }
                        mma16816(sum, H, bp0, bp1);
                        mma16816(sum, H, bl0, bl1);
                        if constexpr (kBits == 10) {
#pragma unroll
                            for (int x2 = 0; x2 < 4; ++x2) acc[mt][x2] += page_sum[x2];
                        }
                    }
                }
            }
            __syncwarp();
            if (lane == 0)   // release the stage to the producer
                asm volatile("mbarrier.arrive.shared::cta.b64 _, [%0];" ::"r"(smem_addr(&empty[s])) : "memory");
        }

        // ---- warp totals for heads 2c, 2c+1 (reduce over the token rows g) ----------------
#pragma unroll
        for (int o = 4; o < 32; o <<= 1)
#pragma unroll
            for (int e = 0; e < 2; ++e) {
                l_part[e] += __shfl_xor_sync(0xffffffffu, l_part[e], o);
                d_part[e] += __shfl_xor_sync(0xffffffffu, d_part[e], o);
                if constexpr (kTierB) db_part[e] += __shfl_xor_sync(0xffffffffu, db_part[e], o);
                if constexpr (kValue) vt_part[e] += __shfl_xor_sync(0xffffffffu, vt_part[e], o);
                spv_part[e] += __shfl_xor_sync(0xffffffffu, spv_part[e], o);
            }
        if constexpr (kValue)
            for (int o = 1; o < 32; o <<= 1) vmax = fmaxf(vmax, __shfl_xor_sync(0xffffffffu, vmax, o));
        const float inv_lam = pow2(lam_exp == INT_MIN ? 0 : -lam_exp);

        // ---- CTA merge over the consumer warps: one partial per segment --------------------
        // (heads hb .. hb + kMergeHeads - 1 at a time)
        constexpr int kMH = Sm::kMergeHeads;
        auto merge_row = [&](int w, int hh) { return mbuf + (w * kMH + hh) * Sm::kMergeRow; };
        auto merge_sums = [&](int w, int hh) {   // m, l, D, Tier-B D, value term, max ||v||
            return Sm::kDense ? mbuf + kWsPairs * kMH * kHeadDim + (w * kMH + hh) * 6 : merge_row(w, hh) + kHeadDim;
        };
#pragma unroll 1
        for (int hb = 0; hb < kMaxGroup; hb += kMH) {
        if (hb >= G) break;
        consumer_sync();   // all consumers are done with their stages and with mbuf's last use
        if (2 * c >= hb && 2 * c < hb + kMH) {
            float* wb = mbuf + pw * kMH * Sm::kMergeRow - hb * Sm::kMergeRow;
#pragma unroll
            for (int e = 0; e < 2; ++e) {
                float* row = wb + (2 * c + e) * Sm::kMergeRow;
                const float add = kKappaV * spv_part[e] * inv_lam;   // spv is in the lam frame
#pragma unroll
                for (int mt = 0; mt < 8; ++mt) {   // m-tile rows g, g + 8: dims 16 mt + g, 16 mt + g + 8
                    row[16 * mt + g] = fmaf(acc[mt][e], inv_lam, add);
                    row[16 * mt + g + 8] = fmaf(acc[mt][e + 2], inv_lam, add);
                }
                if (g == 0) {
                    float* sums = Sm::kDense ? merge_sums(pw, 2 * c + e - hb) : row + kHeadDim;
                    sums[0] = m_run[e];
                    sums[1] = l_part[e];
                    sums[2] = d_part[e];
                    if constexpr (kTierB) sums[3] = db_part[e];
                    if constexpr (kValue) {
                        sums[4] = vt_part[e];
                        sums[5] = vmax;
                    }
                }
            }
        }
        consumer_sync();
        const size_t unit = (size_t)b * p.num_kv_heads + h;
        // flattened plan: share j's segment of sequence b goes to partial h (shares + batch) + j + b
        const int shares = p.splits / p.num_kv_heads;
        const size_t pid = kFlat ? (size_t)h * (shares + p.batch) + blockIdx.x / p.num_kv_heads + b
                                 : unit * p.splits + blockIdx.x;
        float* part_out = p.partials + pid * (kMaxGroup * kPartialStride);
        const int hn = min(kMH, G - hb);
        for (int idx = threadIdx.x; idx < hn * 33; idx += 32 * kWsPairs) {
            const int hh = idx / 33, ch = idx % 33;
            float mw[kWsPairs];
            float M = -INFINITY;
#pragma unroll
            for (int w = 0; w < kWsPairs; ++w) {
                mw[w] = merge_sums(w, hh)[0];
                M = fmaxf(M, mw[w]);
            }
            float4 s4 = make_float4(0.f, 0.f, 0.f, 0.f);
            const int col = (ch < 32) ? 4 * ch : kHeadDim + 1;
#pragma unroll
            for (int w = 0; w < kWsPairs; ++w) {
                if (mw[w] == -INFINITY) continue;   // a warp without pages: its values are not read
                const float wt = fast_exp2(mw[w] - M);
                const float* src = Sm::kDense && ch >= 32 ? merge_sums(w, hh) + 1 : merge_row(w, hh) + col;
                if (ch < 32) {
                    const float4 v = *reinterpret_cast<const float4*>(src);
                    s4.x = fmaf(wt, v.x, s4.x); s4.y = fmaf(wt, v.y, s4.y);
                    s4.z = fmaf(wt, v.z, s4.z); s4.w = fmaf(wt, v.w, s4.w);
                } else {
                    s4.x = fmaf(wt, src[0], s4.x);
                    s4.y = fmaf(wt, src[1], s4.y);
                    if constexpr (kTierB) s4.z = fmaf(wt, src[2], s4.z);
                    if constexpr (kValue) s4.w = fmaf(wt, src[3], s4.w);
                }
            }
            float* dst = part_out + (hb + hh) * kPartialStride;
            if (ch < 32) {
                *reinterpret_cast<float4*>(dst + 4 * ch) = s4;
            } else {
                dst[kHeadDim] = M;
                dst[kHeadDim + 1] = s4.x;
                dst[kHeadDim + 2] = s4.y;
                if constexpr (kTierB) dst[kHeadDim + 3] = s4.z;
                if constexpr (kValue) {
                    float vm = 0.f;
                    for (int w = 0; w < kWsPairs; ++w)
                        vm = fmaxf(vm, merge_sums(w, hh)[5]);
                    dst[kHeadDim + 4] = s4.w;
                    dst[kHeadDim + 5] = vm;
                }
            }
        }
        }
    };
    if constexpr (kFlat) {
        for (bool more = have; more; more = ws_step<kWsPairs>(p, my_seg, lane)) consume(*my_seg);
    } else {
        if (have) consume(sg);
    }
}

// Merge of the per-split partials of one (sequence, query head), 32 output
// dims per CTA: out = sum_s w_s acc_s / sum_s w_s l_s with w_s = 2^(m_s - M),
// D = sum_s w_s D_s / sum_s w_s l_s, meter_raw = D (D + 2) / 2 (§6.2.2: the
// meter accumulator merges under the same LSE weights as the output).  Each
// warp folds its splits with a running maximum in one pass.
constexpr int kMergeWarps = 8;

template <int kX>
__global__ void __launch_bounds__(32 * kMergeWarps) merge_kernel(const __grid_constant__ DecodeParams p) {
    grid_dep_launch();   // the next kernel waits for this grid before reading its outputs
    grid_dep_wait();
    const int chunk = blockIdx.x, hq = blockIdx.y, b = blockIdx.z;
    const int lane = threadIdx.x & 31, warp = threadIdx.x >> 5;
    const int h = hq / p.group, hh = hq % p.group;
    const size_t unit = (size_t)b * p.num_kv_heads + h;
    const int count = p.splits;   // split plan with many splits (otherwise merge_warp_kernel)
    const float* base = p.partials + unit * p.splits * (kMaxGroup * kPartialStride) + hh * kPartialStride;
    const size_t split_stride = kMaxGroup * kPartialStride;
    __shared__ float red[kMergeWarps][38];

    // all of this warp's split rows of a round are loaded before any is
    // combined, so the loads overlap (one memory latency per round, not per split)
    constexpr int kMaxRows = 16;   // rows per warp and round
    constexpr bool tier_b = (kX & kXTierB) != 0, vside = (kX & kXValue) != 0, repair = (kX & kXRepair) != 0;
    float M = -INFINITY, acc = 0.f, L = 0.f, Dn = 0.f, Db = 0.f, Vt = 0.f, Vm = 0.f;
    for (int s0 = warp; s0 < count; s0 += kMergeWarps * kMaxRows) {
        float ms[kMaxRows], v[kMaxRows], ls[kMaxRows], ds[kMaxRows], dbs[kMaxRows], vts[kMaxRows];
#pragma unroll
        for (int i = 0; i < kMaxRows; ++i) {
            const int s = s0 + i * kMergeWarps;
            ms[i] = -INFINITY;
            v[i] = ls[i] = ds[i] = dbs[i] = vts[i] = 0.f;
            if (s < count) {
                const float* ps = base + s * split_stride;
                ms[i] = __ldcg(ps + kHeadDim);
                v[i] = __ldcg(ps + 32 * chunk + lane);
                ls[i] = __ldcg(ps + kHeadDim + 1);
                ds[i] = __ldcg(ps + kHeadDim + 2);
                if (tier_b) dbs[i] = __ldcg(ps + kHeadDim + 3);
                if (vside) {
                    vts[i] = __ldcg(ps + kHeadDim + 4);
                    Vm = fmaxf(Vm, __ldcg(ps + kHeadDim + 5));
                }
            }
        }
        float Mr = M;
#pragma unroll
        for (int i = 0; i < kMaxRows; ++i) Mr = fmaxf(Mr, ms[i]);
        if (Mr == -INFINITY) continue;
        if (Mr > M) {   // move the running sums to the new reference
            const float f = (M == -INFINITY) ? 0.f : fast_exp2(M - Mr);
            acc *= f; L *= f; Dn *= f; Db *= f; Vt *= f;
            M = Mr;
        }
#pragma unroll
        for (int i = 0; i < kMaxRows; ++i) {
            if (ms[i] == -INFINITY) continue;          // empty split: values not read
            const float w = fast_exp2(ms[i] - M);
            acc = fmaf(w, v[i], acc);
            L = fmaf(w, ls[i], L);
            Dn = fmaf(w, ds[i], Dn);
            Db = fmaf(w, dbs[i], Db);
            Vt = fmaf(w, vts[i], Vt);
        }
    }
    red[warp][lane] = acc;
    if (lane == 0) {
        red[warp][32] = M;
        red[warp][33] = L;
        red[warp][34] = Dn;
        red[warp][35] = Db;
        red[warp][36] = Vt;
        red[warp][37] = Vm;
    }
    __syncthreads();
    if (warp == 0) {
        float Mt = -INFINITY;
#pragma unroll
        for (int w = 0; w < kMergeWarps; ++w) Mt = fmaxf(Mt, red[w][32]);
        float a = 0.f, l = 0.f, dn = 0.f, db = 0.f, vt = 0.f, vm = 0.f;
        if (vside)
            for (int w = 0; w < kMergeWarps; ++w) vm = fmaxf(vm, red[w][37]);
        if (Mt != -INFINITY) {
#pragma unroll
            for (int w = 0; w < kMergeWarps; ++w) {
                if (red[w][32] == -INFINITY) continue;
                const float f = fast_exp2(red[w][32] - Mt);
                a = fmaf(f, red[w][lane], a);
                l = fmaf(f, red[w][33], l);
                dn = fmaf(f, red[w][34], dn);
                db = fmaf(f, red[w][35], db);
                vt = fmaf(f, red[w][36], vt);
            }
        }
        const size_t cell = (size_t)b * p.num_q_heads + hq;
        p.out[cell * kHeadDim + 32 * chunk + lane] = l > 0.f ? a / l : 0.f;
        if (chunk == 0 && lane == 0) {
            float raw = 0.f;
            if (l > 0.f) {
                const float D = d_upper(dn / l);        // A - 1, rounded up
                raw = raw_or_inf(0.5f * D * (D + 2.0f));   // (A^2 - 1) / 2, +inf on overflow
            }
            p.meter_raw[cell] = raw;
            p.meter[cell] = fminf(1.0f, raw);
            if (repair) p.softmax_norm[cell] = make_float2(Mt, l);
            if (tier_b) {
                float rb = 0.f;
                if (l > 0.f) {
                    const float D = d_upper(db / l);
                    rb = raw_or_inf(0.5f * D * (D + 2.0f));
                }
                p.meter_b_raw[cell] = rb;
                p.meter_b[cell] = fminf(1.0f, rb);
            }
            if (vside) {   // ||y - y^|| <= 2 TV max ||v|| + sum p~ rho^v, TV <= meter
                const float vterm = l > 0.f ? vt / l * kDRel : 0.f;   // rounded up like D
                p.value_term[cell] = vterm;
                p.v_max[cell] = vm;
                p.out_bound[cell] = 2.0f * fminf(1.0f, raw) * vm + vterm;
            }
        }
    }
}

}  // namespace

// The merge is launched early (programmatic dependent) and its CTAs become
// resident on the SMs the decode grid frees first.  When the merge grid fits
// in one wave, each CTA also reserves more than half of an SM's shared memory
// (unused), so no two share an SM and the merge runs spread over the GPU
// instead of packed onto the first few SMs to free up.
constexpr int kMergeSpreadSmem = 118784;

// Merge where a unit has only a few partials: the flattened plan (its
// sequence's cuts) and a split plan of at most kWarpMergeSplits splits.  kW warps per
// (sequence, query head, 32 output dims) take every kW-th partial with the same
// running-maximum update as merge_kernel and add up through shared memory, so a CTA of 8
// warps serves 8 / kW outputs.  A long sequence in a small batch has up to 38 cuts at 4 KV
// heads, which one warp folds in five rounds of loads: 2 sequences of 984 pages 24.3 us a
// decode with kW = 1, 21.2 with 8, sequences of 1975 and 1 pages 28.3 and 21.9.  A batch of
// many sequences has few cuts each, and more CTAs only start later: 16 sequences of 387
// pages 44.7 us with kW = 1 or 2, 45.8 with 4; 38 of 52 pages 19.4 with 1, 21.3 with 2.
// So kW is the largest of 8, 4, 2, 1 that keeps the launch within 24 warps per SM, the
// three CTAs that fit with the value side's 80 registers (kW = 1, of any size: four).
constexpr int kWarpMergeSplits = 8;

// kHint (flattened plan, at most a sequence per lane): the partials are found from the
// context lengths as they stand before the wait (hints: read past L1).  After it the
// lengths are read again next to the partials, which are folded anew if one has changed.
// 2 sequences of 988 pages: 20.0 -> 18.7 us a decode; 16 of 387: 42.6 -> 41.4.  Larger
// batches and the split plan do without: there the second pass only cost (1000 fp8 sequences
// of 1 to 4 pages, 28 heads: 91.2 us with it, 87.2 without).
template <int kX, int kW, bool kHint>
__global__ void __launch_bounds__(32 * kMergeWarps, kW == 1 ? 4 : 3) merge_warp_kernel(const __grid_constant__ DecodeParams p) {
    grid_dep_launch();   // the next kernel waits for this grid before reading its outputs
    const int lane = threadIdx.x & 31, warp = threadIdx.x >> 5, sub = warp % kW;
    const long long item = (long long)blockIdx.x * (kMergeWarps / kW) + warp / kW;
    const bool live = item < (long long)p.batch * p.num_q_heads * (kHeadDim / 32);   // warp-uniform
    if (kHint && kW == 1 && !live) return;
    int cx = kHint && lane < p.batch ? __ldcg(p.ctx_lens + lane) : 0;
    const int chunk = (int)(item % (kHeadDim / 32));
    const int hq = (int)((item / (kHeadDim / 32)) % p.num_q_heads);
    const int b = (int)(item / ((kHeadDim / 32) * p.num_q_heads));
    const int h = hq / p.group, hh = hq % p.group;
    constexpr bool tier_b = (kX & kXTierB) != 0, vside = (kX & kXValue) != 0, repair = (kX & kXRepair) != 0;

    // A sequence's span in the flattened layout.
    auto span_of = [&](int len) {
        return flat_span((uint32_t)(max(0, min(len, p.max_pages * kPage)) + kPage - 1) / kPage);
    };
    // Flattened plan.  The sequences lie end to end, the n_b > 0 pages of sequence b
    // from P_b on and kCutPages empty positions behind them (lengths clamped, as in the
    // decode); share j of the splits / Hkv shares took positions
    // [j R - off, (j + 1) R - off) in each head, so the unit's segments are those of
    // shares (P_b + off) / R .. (P_b + off + n_b - 1) / R, stored at partials
    // h (shares + batch) + j + b, consecutive.
    int count = 0;
    const float* base = nullptr;
    auto find_flat = [&](uint32_t before, uint32_t total, uint32_t nb) {
        const uint32_t shares = max(1, p.splits / p.num_kv_heads);
        const FlatShares f(total, shares);
        const uint32_t j0 = (before + f.off) / f.R;
        count = nb > 0 ? (int)((before + f.off + nb - 1) / f.R - j0 + 1) : 0;
        base = p.partials + ((size_t)h * (shares + p.batch) + (size_t)(j0 + b)) * (kMaxGroup * kPartialStride) +
               hh * kPartialStride;
    };
    auto find_hinted = [&] {
        if (kW > 1 && !live) return;
        const uint32_t span = lane < p.batch ? span_of(cx) : 0u, own = __shfl_sync(0xffffffffu, span, b);
        find_flat(__reduce_add_sync(0xffffffffu, lane < b ? span : 0u), __reduce_add_sync(0xffffffffu, span),
                  own > 0 ? own - kCutPages : 0u);
    };
    int now = 0;
    if constexpr (kHint) {
        find_hinted();
        grid_dep_wait();
        now = lane < p.batch ? load_dep(p.ctx_lens + lane) : 0;
    } else {
        grid_dep_wait();
        if (p.pages_per_split > 0) {
            // Split plan: the unit's splits are consecutive; those past the
            // sequence's last page hold no pages (their maximum is -inf) and are
            // not read.
            if (!live) return;   // (a warp per output)
            const int nb = (clamped_ctx(p, b) + kPage - 1) / kPage;
            count = min(p.splits, (nb + p.pages_per_split - 1) / p.pages_per_split);
            base = p.partials + ((size_t)b * p.num_kv_heads + h) * p.splits * (kMaxGroup * kPartialStride) +
                   hh * kPartialStride;
        } else {
            // The CTA's threads add up the spans together, up to the sequence of its first
            // output (a scan by every warp: 1000 sequences of 45 pages, 56 heads, 822 us a
            // decode; so 722).
            __shared__ uint32_t sums[2][kMergeWarps];
            const int b0 = (int)((long long)blockIdx.x * (kMergeWarps / kW) / ((kHeadDim / 32) * p.num_q_heads));
            uint32_t before = 0, total = 0;
            for (int i = threadIdx.x; i < p.batch; i += 32 * kMergeWarps) {
                const uint32_t span = span_of(load_dep(p.ctx_lens + i));
                total += span;
                if (i < b0) before += span;
            }
            total = __reduce_add_sync(0xffffffffu, total);
            before = __reduce_add_sync(0xffffffffu, before);
            if (lane == 0) {
                sums[0][warp] = before;
                sums[1][warp] = total;
            }
            __syncthreads();
            if (kW == 1 && !live) return;
            if (live) {
                before = __reduce_add_sync(0xffffffffu, lane < kMergeWarps ? sums[0][lane] : 0u);
                total = __reduce_add_sync(0xffffffffu, lane < kMergeWarps ? sums[1][lane] : 0u);
                for (int i = b0; i < b; ++i) before += span_of(load_dep(p.ctx_lens + i));
                find_flat(before, total, (uint32_t)(clamped_ctx(p, b) + kPage - 1) / kPage);
            }
        }
    }
    constexpr int kRows = 8;   // rows loaded per round before any is combined
    float M = -INFINITY, acc = 0.f, L = 0.f, Dn = 0.f, Db = 0.f, Vt = 0.f, Vm = 0.f;
    for (bool again = kHint;; again = false) {
        for (int s0 = sub; s0 < count; s0 += kRows * kW) {
            float ms[kRows], v[kRows], ls[kRows], ds[kRows], dbs[kRows], vts[kRows];
#pragma unroll
            for (int i = 0; i < kRows; ++i) {
                ms[i] = -INFINITY;
                v[i] = ls[i] = ds[i] = dbs[i] = vts[i] = 0.f;
                if (s0 + i * kW < count) {
                    const float* ps = base + (size_t)(s0 + i * kW) * (kMaxGroup * kPartialStride);
                    ms[i] = __ldcg(ps + kHeadDim);
                    v[i] = __ldcg(ps + 32 * chunk + lane);
                    ls[i] = __ldcg(ps + kHeadDim + 1);
                    ds[i] = __ldcg(ps + kHeadDim + 2);
                    if (tier_b) dbs[i] = __ldcg(ps + kHeadDim + 3);
                    if (vside) {
                        vts[i] = __ldcg(ps + kHeadDim + 4);
                        Vm = fmaxf(Vm, __ldcg(ps + kHeadDim + 5));
                    }
                }
            }
            float Mr = M;
#pragma unroll
            for (int i = 0; i < kRows; ++i) Mr = fmaxf(Mr, ms[i]);
            if (Mr == -INFINITY) continue;
            if (Mr > M) {
                const float f = (M == -INFINITY) ? 0.f : fast_exp2(M - Mr);
                acc *= f; L *= f; Dn *= f; Db *= f; Vt *= f;
                M = Mr;
            }
#pragma unroll
            for (int i = 0; i < kRows; ++i) {
                if (ms[i] == -INFINITY) continue;
                const float w = fast_exp2(ms[i] - M);
                acc = fmaf(w, v[i], acc);
                L = fmaf(w, ls[i], L);
                Dn = fmaf(w, ds[i], Dn);
                Db = fmaf(w, dbs[i], Db);
                Vt = fmaf(w, vts[i], Vt);
            }
        }
        if (!again || !__any_sync(0xffffffffu, now != cx)) break;
        cx = now;
        find_hinted();
        M = -INFINITY;
        acc = L = Dn = Db = Vt = Vm = 0.f;
    }
    if constexpr (kW > 1) {
        __shared__ float red[kMergeWarps][38];
        red[warp][lane] = acc;
        if (lane == 0) {
            red[warp][32] = M;
            red[warp][33] = L;
            red[warp][34] = Dn;
            red[warp][35] = Db;
            red[warp][36] = Vt;
            red[warp][37] = Vm;
        }
        __syncthreads();
        if (!live || sub != 0) return;
#pragma unroll
        for (int w = 1; w < kW; ++w) {
            M = fmaxf(M, red[warp + w][32]);
            Vm = fmaxf(Vm, red[warp + w][37]);
        }
        acc = L = Dn = Db = Vt = 0.f;
        if (M != -INFINITY) {
#pragma unroll
            for (int w = 0; w < kW; ++w) {
                const float* r = red[warp + w];
                if (r[32] == -INFINITY) continue;
                const float f = fast_exp2(r[32] - M);
                acc = fmaf(f, r[lane], acc);
                L = fmaf(f, r[33], L);
                Dn = fmaf(f, r[34], Dn);
                Db = fmaf(f, r[35], Db);
                Vt = fmaf(f, r[36], Vt);
            }
        }
    }
    const size_t cell = (size_t)b * p.num_q_heads + hq;
    p.out[cell * kHeadDim + 32 * chunk + lane] = L > 0.f ? acc / L : 0.f;
    if (chunk == 0 && lane == 0) {
        float raw = 0.f;
        if (L > 0.f) {
            const float D = d_upper(Dn / L);
            raw = raw_or_inf(0.5f * D * (D + 2.0f));
        }
        p.meter_raw[cell] = raw;
        p.meter[cell] = fminf(1.0f, raw);
        if (repair) p.softmax_norm[cell] = make_float2(M, L);
        if (tier_b) {
            float rb = 0.f;
            if (L > 0.f) {
                const float D = d_upper(Db / L);
                rb = raw_or_inf(0.5f * D * (D + 2.0f));
            }
            p.meter_b_raw[cell] = rb;
            p.meter_b[cell] = fminf(1.0f, rb);
        }
        if (vside) {
            const float vterm = L > 0.f ? Vt / L * kDRel : 0.f;
            p.value_term[cell] = vterm;
            p.v_max[cell] = Vm;
            p.out_bound[cell] = 2.0f * fminf(1.0f, raw) * Vm + vterm;
        }
    }
}

template <int kX>
static cudaError_t launch_merge(const DecodeParams& p, cudaStream_t stream) {
    static PerDevice<int, cudaError_t> state;
    int num_sms = 0;   // 0: the spread request is not used
    (void)per_device(state, num_sms, [](int& sms) {
        int dev = 0, n = 0;
        sms = 0;
        if (cudaGetDevice(&dev) == cudaSuccess &&
            cudaDeviceGetAttribute(&n, cudaDevAttrMultiProcessorCount, dev) == cudaSuccess &&
            cudaFuncSetAttribute(merge_kernel<kX>, cudaFuncAttributeMaxDynamicSharedMemorySize, kMergeSpreadSmem) ==
                cudaSuccess)
            sms = n;
        (void)cudaFuncSetAttribute(merge_kernel<kX>, cudaFuncAttributePreferredSharedMemoryCarveout,
                                   (int)cudaSharedmemCarveoutMaxShared);
        (void)cudaGetLastError();   // a refused hint leaves no sticky error behind
        return cudaSuccess;
    });
    if (p.pages_per_split == 0 || p.splits <= kWarpMergeSplits) {   // a few partials per unit
        const long items = (long)p.batch * p.num_q_heads * (kHeadDim / 32), room = 24L * num_sms;
        auto go = [&](auto kernel, int w) {
            const long per = kMergeWarps / w;
            return launch_pdl(kernel, dim3((unsigned)((items + per - 1) / per)), dim3(32 * kMergeWarps), 0, stream, p);
        };
        const bool flat = p.pages_per_split == 0;
        const int w = !flat ? 1 : items * 8 <= room ? 8 : items * 4 <= room ? 4 : items * 2 <= room ? 2 : 1;
        if (flat && p.batch <= 32)
            return w == 8   ? go(merge_warp_kernel<kX, 8, true>, 8)
                   : w == 4 ? go(merge_warp_kernel<kX, 4, true>, 4)
                   : w == 2 ? go(merge_warp_kernel<kX, 2, true>, 2)
                            : go(merge_warp_kernel<kX, 1, true>, 1);
        return w == 8   ? go(merge_warp_kernel<kX, 8, false>, 8)
               : w == 4 ? go(merge_warp_kernel<kX, 4, false>, 4)
               : w == 2 ? go(merge_warp_kernel<kX, 2, false>, 2)
                        : go(merge_warp_kernel<kX, 1, false>, 1);
    }
    const dim3 grid(kHeadDim / 32, p.num_q_heads, p.batch);
    const long ctas = (long)grid.x * grid.y * grid.z;
    const size_t smem = (num_sms > 0 && ctas <= num_sms) ? kMergeSpreadSmem : 0;
    return launch_pdl(merge_kernel<kX>, grid, dim3(32 * kMergeWarps), smem, stream, p);
}

cudaError_t launch_merge_x(const DecodeParams& p, int x, cudaStream_t stream) {
    return x == kXTierB ? launch_merge<kXTierB>(p, stream)
         : x == kXValue ? launch_merge<kXValue>(p, stream)
         : x == kXRepair ? launch_merge<kXRepair>(p, stream) : launch_merge<0>(p, stream);
}

template <bool kInt8, int kX>
static cudaError_t launch_two_per_sm(const DecodeParams& p, cudaStream_t stream) {
    static PerDevice<Configured, cudaError_t> configured;
    constexpr int kSmem = TwoPerSm<kInt8, kX>::kSmemBytes;
    if (cudaError_t e = configure(configured, decode_kernel<kInt8, kX>, kSmem)) return e;
    DkParams dp;
    dp.p = p;
    if (!encode_page_map(&dp.k_map, p.k_codes, p.num_pages, p.num_kv_heads) ||
        !encode_page_map(&dp.v_map, p.v_codes, p.num_pages, p.num_kv_heads))
        return cudaErrorInvalidValue;
    const dim3 grid(p.splits, p.num_kv_heads, p.batch);
    cudaError_t e = launch_pdl(decode_kernel<kInt8, kX>, grid, dim3(kThreads), kSmem, stream, dp);
    if (e != cudaSuccess) return e;
    // the merge is a programmatic dependent too: its CTAs are scheduled while
    // the decode grid drains and wait (griddepcontrol.wait) for all of it
    return launch_merge<kX>(p, stream);
}

// cuTensorMapEncodeTiled through the runtime's driver entry point (the
// library does not link the driver library itself).
static PFN_cuTensorMapEncodeTiled_v12000 tensor_map_encoder() {
    static std::once_flag once;
    static PFN_cuTensorMapEncodeTiled_v12000 fn = nullptr;
    std::call_once(once, [] {
        void* f = nullptr;
        cudaDriverEntryPointQueryResult q;
        if (cudaGetDriverEntryPointByVersion("cuTensorMapEncodeTiled", &f, 12000, cudaEnableDefault, &q) ==
                cudaSuccess &&
            q == cudaDriverEntryPointSuccess)
            fn = reinterpret_cast<PFN_cuTensorMapEncodeTiled_v12000>(f);
    });
    return fn;
}

// One layer's code array [num_pages][Hkv][16][128] bytes as a 3-D tensor
// (channel, slot, page * Hkv + head); a box is one page of one head, written
// to shared memory with the 128-byte swizzle.
bool encode_page_map(CUtensorMap* map, const void* codes, int num_pages, int num_kv_heads) {
    PFN_cuTensorMapEncodeTiled_v12000 enc = tensor_map_encoder();
    if (!enc) return false;
    const cuuint64_t dims[3] = {(cuuint64_t)kHeadDim, (cuuint64_t)kPage, (cuuint64_t)num_pages * num_kv_heads};
    const cuuint64_t strides[2] = {(cuuint64_t)kHeadDim, (cuuint64_t)kHeadDim * kPage};
    const cuuint32_t box[3] = {(cuuint32_t)kHeadDim, (cuuint32_t)kPage, 1};
    const cuuint32_t elem[3] = {1, 1, 1};
    return enc(map, CU_TENSOR_MAP_DATA_TYPE_UINT8, 3, const_cast<void*>(codes), dims, strides, box, elem,
               CU_TENSOR_MAP_INTERLEAVE_NONE, CU_TENSOR_MAP_SWIZZLE_128B, CU_TENSOR_MAP_L2_PROMOTION_L2_256B,
               CU_TENSOR_MAP_FLOAT_OOB_FILL_NONE) == CUDA_SUCCESS;
}

template <int kBits, int kX>
static cudaError_t launch_ws(const DecodeParams& p, cudaStream_t stream) {
    constexpr int kSmem = WsSmem<kBits, (kX & kXFlat) != 0>::kBytes;
    static PerDevice<Configured, cudaError_t> configured;
    if (cudaError_t e = configure(configured, decode_ws_kernel<kBits, kX>, kSmem)) return e;
    WsParams wp;
    wp.p = p;
    if constexpr ((kX & kXAppend) != 0) {   // the cache as the write path sees it
        WriteParams& w = wp.w;
        w.k = w.v = nullptr;
        w.slot_mapping = p.slot_new;
        w.k_codes = const_cast<uint8_t*>(p.k_codes);
        w.v_codes = const_cast<uint8_t*>(p.v_codes);
        w.k_scale = const_cast<__half*>(p.k_scale);
        w.v_scale = const_cast<__half*>(p.v_scale);
        w.k_witness = const_cast<__half*>(p.k_witness);
        w.v_witness = nullptr;
        w.dev_status = p.status;
        w.n_tok = p.batch;
        w.num_kv_heads = p.num_kv_heads;
        w.num_pages = p.num_pages;
        w.layer = p.layer;
        w.rope_layout = p.rope_layout;
        w.keys = p.keys;
    }
    if (!encode_page_map(&wp.k_map, p.k_codes, p.num_pages, p.num_kv_heads) ||
        !encode_page_map(&wp.v_map, p.v_codes, p.num_pages, p.num_kv_heads))
        return cudaErrorInvalidValue;
    const bool flat = p.pages_per_split == 0;
    const dim3 grid = flat ? dim3(p.splits, 1, 1) : dim3(p.splits, p.num_kv_heads, p.batch);
    cudaError_t e = launch_pdl(decode_ws_kernel<kBits, kX>, grid, dim3(kWsThreads), kSmem, stream, wp);
    if (e != cudaSuccess) return e;
    return launch_merge<kX & ~(kXAppend | kXFlat | kXStall)>(p, stream);
}

template <int kBits, int kF>
static cudaError_t launch_ws_x(const DecodeParams& p, int x, cudaStream_t stream) {
    if constexpr (kBits == 8)
        if (x == kXAppend) return launch_ws<8, kXAppend | kF>(p, stream);
    return x == kXTierB  ? launch_ws<kBits, kXTierB | kF>(p, stream)
         : x == kXValue  ? launch_ws<kBits, kXValue | kF>(p, stream)
         : x == kXRepair ? launch_ws<kBits, kXRepair | kF>(p, stream) : launch_ws<kBits, kF>(p, stream);
}

cudaError_t launch_decode(const DecodeParams& p, int scheme, int bits, cudaStream_t stream) {
    if (p.batch == 0) return cudaSuccess;
    if (scheme == WC_SCHEME_DITHER_INT8_G32) return launch_decode_g32(p, stream);
    // Tier B (dithered INT8 only), the value side and the repair terms are
    // requested by separate entry points, never together (checked by the caller)
    const int x = (p.meter_b ? kXTierB : 0) | (p.value_term ? kXValue : 0) | (p.page_terms ? kXRepair : 0) |
                  (p.k_new ? kXAppend : 0);
    const bool flat = p.pages_per_split == 0;
    if (scheme == WC_SCHEME_FP8_E4M3)   // always the split plan (plan_decode)
        return flat           ? cudaErrorNotSupported
             : x == kXValue  ? launch_two_per_sm<false, kXValue>(p, stream)
             : x == kXRepair ? launch_two_per_sm<false, kXRepair>(p, stream) : launch_two_per_sm<false, 0>(p, stream);
    if (p.two_per_sm)                   // 10-bit dither, split plan (plan_decode)
        return flat || bits != 10    ? cudaErrorNotSupported
             : x == kXTierB  ? launch_two_per_sm<true, kXTierB>(p, stream)
             : x == kXValue  ? launch_two_per_sm<true, kXValue>(p, stream)
             : x == kXRepair ? launch_two_per_sm<true, kXRepair>(p, stream) : launch_two_per_sm<true, 0>(p, stream);
    if (p.stall_page >= 0)   // failure-detection test (checked by the caller: 8-bit dither, no extras)
        return bits == 8 && !flat && x == 0 ? launch_ws<8, kXStall>(p, stream) : cudaErrorNotSupported;
    if (bits == 8) return flat ? launch_ws_x<8, kXFlat>(p, x, stream) : launch_ws_x<8, 0>(p, x, stream);
    return flat ? launch_ws_x<10, kXFlat>(p, x, stream) : launch_ws_x<10, 0>(p, x, stream);
}

}  // namespace wc
