// Write path: quantize post-RoPE K/V rows into the paged cache and store the
// K band-norm residual witness (§6.2.1 write kernel; §4.1 Eq. witness;
// §4.2 subtractive dither).
//
// A warp handles four (token, KV head) units, their K rows and then their V rows (few
// units: one of the two), 8 lanes per row.  Each lane owns 16 consecutive channels, so it
// loads 32 B of fp16, stores 16 B of codes, and (for the dither schemes) consumes exactly
// one Philox4x32-10 call per row and 16 channels.
//
// Grouped scheme (§6.2.3 "Storage side" and §6.2.5 "Fixed-channel outlier bypass"):
// one fp16 scale per 32-channel group (a lane pair), the group amax leaving
// out the bypassed channels of the KV head's fixed RoPE pairs, which are
// stored exactly (fp16, code 0).  A row is stored in a permuted channel order
// with the dither drawn by storage position; storage position p holds channel
//   K:  16 ((p >> 2) & 7) + 4 (p >> 5) + (p & 3)
//   V:  16 ((p >> 1) & 7) + 8 (p & 1) + (p >> 4)
// (the decode's fragment order: each QK k-step and each PV m-tile then meets
// one group).  The lane's Philox call covers storage positions 16 sub .. +15;
// dither bytes and codes move between storage and channel order through a
// 128-byte shared row per unit, so quantization runs in channel order.
#include <cooperative_groups.h>

#include "dispatch.h"
#include "write_row.cuh"

namespace cg = cooperative_groups;

namespace wc {

namespace {

// A warp's tasks (rows of 4 units), whose loads are all issued before any is used: more
// bytes in flight per SM.  The K and the V rows of the same units: the row routine is
// then specialised for each, and their Philox calls share the products that do not see
// the tag.  A write of a few tokens takes one task per warp (K rows in warps 0 and 2, V
// rows in 1 and 3): there one row's latency is what counts.  Measured at 32768 x 4 tokens
// and heads against K and V rows in separate warps (us): 8-bit dither 30.4 -> 26.5, 10-bit
// 39.7 -> 35.6, fp8 17.6 -> 15.1, grouped with its packed pass 53.4 -> 44.3.
constexpr int write_units_per_cta(int tasks) { return 2 * 4 * tasks; }

// Two ways of cutting the units (token, KV head) into 4-unit tasks:
//  kPerHead: grid (token groups, Hkv), a task = 4 consecutive tokens of one
//            head, so a warp's code, scale and witness stores are contiguous
//            runs of consecutive slots (prefill);
//  else:     one index over units u = token * Hkv + h, a task = 4 consecutive
//            units, K or V, so a one-token write of up to 8 KV heads is a single CTA
//            (decode steps, where every SM the next decode needs counts).
// Resident CTAs per SM the register budget is sized for, the best of 5 .. 9 in each case
// (at 32768 x 4): 8-bit dither seven at 72 registers (six 6% slower, eight, with 36 bytes of
// spill, 5%), 10-bit six (seven 2% slower), grouped six with 56 bytes of spill (seven, with 84,
// 0.5% faster, but the 2047 x 8 write 10% slower), fp8 eight (ten 3% slower).  One
// task per warp: seven, so that the small writes that take it are one wave (1000 x 8: grouped
// 5.6, six 6.3).
__host__ __device__ constexpr int write_min_blocks(int scheme, int bits, int tasks) {
    return scheme == WC_SCHEME_FP8_E4M3 ? 8 : tasks == 2 && (scheme == WC_SCHEME_DITHER_INT8_G32 || bits == 10) ? 6 : 7;
}
// A write's rows, slots and pair set through the read-only path: 32768 x 4 tokens and heads take 26.6
// us so, 26.9 by ordinary loads (grouped 44.4 and 45.5).  Volatile with a memory clobber, as an
// intrinsic is not: they stay behind the wait, before which this grid reads none of them (the
// prefetch goes to L2).
__device__ __forceinline__ uint4 load_once(const uint4* p) {
    uint4 v;
    asm volatile("ld.global.nc.v4.u32 {%0, %1, %2, %3}, [%4];"
                 : "=r"(v.x), "=r"(v.y), "=r"(v.z), "=r"(v.w) : "l"(p) : "memory");
    return v;
}
__device__ __forceinline__ int load_once(const int32_t* p) {
    int v;
    asm volatile("ld.global.nc.u32 %0, [%1];" : "=r"(v) : "l"(p) : "memory");
    return v;
}

template <int kScheme, int kBits, bool kPerHead, int kTasks>
__global__ void __launch_bounds__(128, write_min_blocks(kScheme, kBits, kTasks)) write_kernel(const __grid_constant__ WriteParams p) {
    constexpr bool kGrouped = kScheme == WC_SCHEME_DITHER_INT8_G32;
    __shared__ __align__(16) uint8_t xrows[kGrouped ? 4 * 4 * kXRowStride : 16];   // [warp][unit][row]
    __shared__ BypassTable btab;
    grid_dep_launch();    // a dependent decode may be scheduled now: it waits for this whole grid
    if constexpr (kPerHead) grid_dep_wait();   // inputs may come from the preceding kernel
    const int lane = threadIdx.x & 31, warp = threadIdx.x >> 5;
    const BypassTable* tab = nullptr;
    if constexpr (kGrouped && kPerHead) {   // one KV head per CTA: its bypass set, once
        if (threadIdx.x < kHeadDim) btab.entry[threadIdx.x] = -1;
        if (threadIdx.x < 4) btab.mask[threadIdx.x] = 0u;
        if (threadIdx.x == 0) btab.bad = 0u;
        __syncthreads();
        if (threadIdx.x < p.num_bypass) {
            const int t = threadIdx.x;
            const int32_t* pr = p.bypass_pairs + (size_t)blockIdx.y * p.num_bypass;
            const int j = load_once(pr + t);
            bool dup = false;   // a pair listed again is ignored after its first occurrence
            for (int u = 0; u < t; ++u) dup = dup || load_once(pr + u) == j;
            if (j < 0 || j >= kHeadDim / 2 || dup) {
                atomicOr(&btab.bad, 1u << t);
                if (p.dev_status) atomicOr(p.dev_status, WC_DEV_BAD_PAIR);
            } else {
                const int a = p.rope_layout == WC_ROPE_HALF ? j : 2 * j;
                const int b = p.rope_layout == WC_ROPE_HALF ? j + kHeadDim / 2 : 2 * j + 1;
                btab.entry[a] = (int8_t)(2 * t);
                btab.entry[b] = (int8_t)(2 * t + 1);
                atomicOr(&btab.mask[a >> 5], 1u << (a & 31));
                atomicOr(&btab.mask[b >> 5], 1u << (b & 31));
            }
        }
        __syncthreads();
        tab = &btab;
    }
    // lanes 8i .. 8i+7 own unit i of the warp's four
    const int sub = lane & 7;                                                  // 16-channel chunk
    const int idx = kTasks == 1 ? (blockIdx.x * 2 + (warp >> 1)) * 4 + (lane >> 3)
                                : (blockIdx.x * 4 + warp) * 4 + (lane >> 3);   // a token (kPerHead) or a unit
    const int n_first = kPerHead ? p.n_tok : p.n_tok * p.num_kv_heads;
    const bool live = idx < n_first;
    if (!__any_sync(0xffffffffu, live)) return;   // warp-uniform: a warp past the end
    int tok = 0, h = 0;
    if (live) {
        if (kPerHead) {
            tok = idx;
            h = blockIdx.y;
        } else {
            tok = idx / p.num_kv_heads;
            h = idx - tok * p.num_kv_heads;
        }
    }
    auto row_src = [&](int row) {   // 0 = K, 1 = V
        return reinterpret_cast<const uint4*>((row == 0 ? p.k : p.v) + ((size_t)tok * p.num_kv_heads + h) * kHeadDim +
                                              sub * 16);
    };
    if constexpr (!kPerHead) {   // a decode step's write: its rows reach L2 while the preceding kernel drains
        if (live) prefetch_l2(row_src(warp & 1));
        grid_dep_wait();
    }
    const int slot = live ? load_once(p.slot_mapping + tok) : -1;
    uint4 raw[kTasks][2];
#pragma unroll
    for (int t = 0; t < kTasks; ++t) {
        const int row = kTasks == 1 ? (warp & 1) : t;
        raw[t][0] = raw[t][1] = make_uint4(0, 0, 0, 0);
        if (live) {
            const uint4* src = row_src(row);
            raw[t][0] = load_once(src);
            raw[t][1] = load_once(src + 1);
        }
    }
    uint8_t* xrow = kGrouped ? xrows + (warp * 4 + (lane >> 3)) * kXRowStride : nullptr;
    if constexpr (kTasks == 1) {
        write_row<kScheme, kBits>(p, raw[0], slot, live, h, warp & 1, sub, xrow, tab);
    } else {
        // 8-bit dither: the two rows' Philox calls advanced together
        uint4 w[2];
        constexpr bool kPre = kScheme != WC_SCHEME_FP8_E4M3 && kBits == 8;
        if constexpr (kPre)
            philox_rows((uint32_t)max(slot, 0), (uint32_t)p.layer * 65536u + (uint32_t)h, (uint32_t)sub, p.keys, w[0], w[1]);
        write_row<kScheme, kBits>(p, raw[0], slot, live, h, 0, sub, xrow, tab, kPre ? &w[0] : nullptr);
        write_row<kScheme, kBits>(p, raw[kTasks - 1], slot, live, h, 1, sub, xrow, tab, kPre ? &w[1] : nullptr);
    }
}

// Bypass-pair calibration: a cluster of 8 CTAs of 32 warps per KV head, or of 16 CTAs of 8
// warps.  Either way 256 chains: chain 32 r + c sums rows 32 r + c + 256 i, and the 32
// chains of an r are added in the order of c.  The narrow cluster gives a chain to a warp:
// one 256-byte row per warp load, lane l squaring channels 4l .. 4l + 3.  In the wide one
// rank r takes the channels 0 .. 63 and rank r + 8 the channels 64 .. 127, and a warp load
// covers the half rows of four chains, 16 bytes a lane.  Rank 0 adds the sums of the eight
// r (distributed shared memory, r's order), adds channels into pairs, and selects a pair
// iff fewer than m pairs rank above it (larger energy, or equal energy and a lower index).
// Both clusters add the same numbers in the same order.  Bytes in flight bound the narrow
// one (4 loads a warp: 32 KB an SM, 1.8 TB/s over 32 SMs); the wide one keeps 64 KB an SM in
// a ring of asynchronous copies on twice the SMs, as deeper batches of loads into registers
// were split up again by the compiler (8.7).  16384 rows x 4 heads: 9.3 -> 6.0 us.
constexpr int kSelPairRing = 16;   // wide: copies in flight per lane

__device__ __forceinline__ void copy16_or_zero(uint4* dst, const __half* src, bool valid) {
    asm volatile("cp.async.cg.shared.global [%0], [%1], 16, %2;\n\tcp.async.commit_group;"
                 :: "r"((uint32_t)__cvta_generic_to_shared(dst)), "l"(src), "r"(valid ? 16 : 0)
                 : "memory");
}

template <bool kWide>
__global__ void __launch_bounds__(kWide ? 256 : 1024)
    select_pairs_kernel(const __half* __restrict__ k, int n_tok, int num_kv_heads, int rope_layout, int m,
                        int32_t* __restrict__ pairs) {
    constexpr int kWidth = kWide ? kHeadDim / 2 : kHeadDim;   // channels of a CTA
    __shared__ float part[32][kHeadDim];
    __shared__ float energy[kHeadDim / 2];
    __shared__ int chosen[kHeadDim / 2];
    cg::cluster_group cluster = cg::this_cluster();
    const int rank = (int)cluster.block_rank();
    const int h = blockIdx.y, tid = threadIdx.x, lane = tid & 31, warp = tid >> 5;
    if constexpr (kWide) {
        const size_t stride = (size_t)num_kv_heads * kHeadDim;
        const int chain = 4 * warp + (lane >> 3), c0 = 8 * (lane & 7);
        const __half* src = k + (size_t)h * kHeadDim + (rank >> 3) * kWidth + c0;
        float a[8] = {0.f, 0.f, 0.f, 0.f, 0.f, 0.f, 0.f, 0.f};
        auto add = [&](uint4 w) {
            const uint32_t ww[4] = {w.x, w.y, w.z, w.w};
#pragma unroll
            for (int i = 0; i < 4; ++i) {
                const float2 f = __half22float2(*reinterpret_cast<const __half2*>(&ww[i]));
                a[2 * i] = fmaf(f.x, f.x, a[2 * i]);
                a[2 * i + 1] = fmaf(f.y, f.y, a[2 * i + 1]);
            }
        };
        extern __shared__ uint4 ring[];   // [kSelPairRing][256]: every thread its own 16 bytes
        uint4* slot = ring + tid;
        const int steps = (n_tok + 255) / 256;
        int t = (rank & 7) * 32 + chain;   // row of the next copy
        for (int i = 0; i < kSelPairRing; ++i, t += 256) copy16_or_zero(slot + 256 * i, t < n_tok ? src + t * stride : k, t < n_tok);
#pragma unroll 1
        for (int s = 0; s < steps; s += kSelPairRing) {
#pragma unroll
            for (int i = 0; i < kSelPairRing; ++i, t += 256) {
                asm volatile("cp.async.wait_group %0;" ::"n"(kSelPairRing - 1) : "memory");
                const uint4 w = slot[256 * i];
                __syncwarp();   // the read stands before the copy into the same slot
                add(w);         // + 0 past the end
                copy16_or_zero(slot + 256 * i, t < n_tok ? src + t * stride : k, t < n_tok);
            }
        }
        asm volatile("cp.async.wait_all;" ::: "memory");
#pragma unroll
        for (int i = 0; i < 8; ++i) part[chain][c0 + i] = a[i];
    } else {
        float a0 = 0.f, a1 = 0.f, a2 = 0.f, a3 = 0.f;
#pragma unroll 4
        for (int t = rank * 32 + warp; t < n_tok; t += 256) {
            const uint2 w = load_dep(reinterpret_cast<const uint2*>(k + ((size_t)t * num_kv_heads + h) * kHeadDim) + lane);
            const float2 f01 = __half22float2(*reinterpret_cast<const __half2*>(&w.x));
            const float2 f23 = __half22float2(*reinterpret_cast<const __half2*>(&w.y));
            a0 = fmaf(f01.x, f01.x, a0);
            a1 = fmaf(f01.y, f01.y, a1);
            a2 = fmaf(f23.x, f23.x, a2);
            a3 = fmaf(f23.y, f23.y, a3);
        }
        part[warp][4 * lane] = a0;
        part[warp][4 * lane + 1] = a1;
        part[warp][4 * lane + 2] = a2;
        part[warp][4 * lane + 3] = a3;
    }
    __syncthreads();
    if (tid < kWidth) {   // this CTA's channel sums in a fixed order (each thread its own column)
        float e = 0.f;
        for (int w = 0; w < 32; ++w) e += part[w][tid];
        part[0][tid] = e;
    }
    cluster.sync();   // every CTA's sums are in its row 0
    if (rank == 0) {
        if (tid < kHeadDim) {
            float e = 0.f;
            for (int r = 0; r < 8; ++r)
                e += cluster.map_shared_rank(&part[0][0], tid / kWidth * 8 + r)[tid % kWidth];
            part[1][tid] = e;
        }
        __syncthreads();
        const int j = tid;
        if (j < kHeadDim / 2) {
            const int a = rope_layout == WC_ROPE_HALF ? j : 2 * j;
            const int b = rope_layout == WC_ROPE_HALF ? j + kHeadDim / 2 : 2 * j + 1;
            energy[j] = part[1][a] + part[1][b];
        }
        __syncthreads();
        if (j < kHeadDim / 2) {
            const float e = energy[j];
            int rnk = 0;
            for (int i = 0; i < kHeadDim / 2; ++i) rnk += (energy[i] > e || (energy[i] == e && i < j)) ? 1 : 0;
            chosen[j] = rnk < m;
        }
        __syncthreads();
        if (j < kHeadDim / 2 && chosen[j]) {
            int pos = 0;
            for (int i = 0; i < j; ++i) pos += chosen[i];
            if (pos < m) pairs[(size_t)h * m + pos] = j;   // NaN energies can make more than m ranks fall below m
        }
    }
    cluster.sync();   // the other CTAs' shared memory stays alive until rank 0 has read it
}

}  // namespace

template <bool kWide>
static cudaError_t launch_pairs(const __half* k, int n_tok, int num_kv_heads, int rope_layout, int m, int32_t* pairs,
                                cudaStream_t stream, int* resident = nullptr) {   // resident: asked instead of a launch
    cudaLaunchConfig_t cfg = {};
    cfg.gridDim = dim3(kWide ? 16 : 8, num_kv_heads);
    cfg.blockDim = dim3(kWide ? 256 : 1024);
    cfg.dynamicSmemBytes = kWide ? kSelPairRing * 256 * 16 : 0;
    cfg.stream = stream;
    cudaLaunchAttribute attr[1];
    attr[0].id = cudaLaunchAttributeClusterDimension;
    attr[0].val.clusterDim.x = cfg.gridDim.x;
    attr[0].val.clusterDim.y = attr[0].val.clusterDim.z = 1;
    cfg.attrs = attr;
    cfg.numAttrs = 1;
    if (resident) return cudaOccupancyMaxActiveClusters(resident, select_pairs_kernel<kWide>, &cfg);
    return cudaLaunchKernelEx(&cfg, select_pairs_kernel<kWide>, k, n_tok, num_kv_heads, rope_layout, m, pairs);
}

// Wide clusters resident at once on the current device; 0 where they cannot be launched.
static int wide_pair_clusters() {
    static PerDevice<int, cudaError_t> state;
    int n = 0;
    const cudaError_t known = per_device(state, n, [](int& clusters) {
        auto kernel = select_pairs_kernel<true>;
        clusters = 0;
        if (cudaFuncSetAttribute(kernel, cudaFuncAttributeNonPortableClusterSizeAllowed, 1) != cudaSuccess ||   // above 8
            cudaFuncSetAttribute(kernel, cudaFuncAttributeMaxDynamicSharedMemorySize, kSelPairRing * 256 * 16) != cudaSuccess ||
            launch_pairs<true>(nullptr, 0, 1, WC_ROPE_HALF, 0, nullptr, nullptr, &clusters) != cudaSuccess) {
            clusters = 0;
            (void)cudaGetLastError();   // the narrow cluster serves instead
        }
        return cudaSuccess;
    });
    return known == cudaSuccess ? n : 0;
}

cudaError_t launch_select_pairs(const __half* k, int n_tok, int num_kv_heads, int rope_layout, int m, int32_t* pairs,
                                cudaStream_t stream) {
    const bool wide = pairs_wide(n_tok, ((uintptr_t)k & 15) == 0, num_kv_heads,
                                 n_tok >= kWidePairRows ? wide_pair_clusters() : 0);
    return wide ? launch_pairs<true>(k, n_tok, num_kv_heads, rope_layout, m, pairs, stream)
                : launch_pairs<false>(k, n_tok, num_kv_heads, rope_layout, m, pairs, stream);
}

cudaError_t launch_write(const WriteParams& p, int scheme, int bits, cudaStream_t stream) {
    if (p.n_tok == 0) return cudaSuccess;
    static PerDevice<Configured, cudaError_t> configured;   // same carveout as the decode kernels: no L1/shared reconfiguration
    Configured c;
    const cudaError_t set = per_device(configured, c, [](Configured&) {
        const void* fns[10] = {(const void*)write_kernel<WC_SCHEME_FP8_E4M3, 8, false, 1>,
                               (const void*)write_kernel<WC_SCHEME_DITHER_INT8, 8, false, 1>,
                               (const void*)write_kernel<WC_SCHEME_DITHER_INT8, 10, false, 1>,
                               (const void*)write_kernel<WC_SCHEME_DITHER_INT8_G32, 8, false, 1>,
                               (const void*)write_kernel<WC_SCHEME_FP8_E4M3, 8, true, 2>,
                               (const void*)write_kernel<WC_SCHEME_DITHER_INT8, 8, true, 2>,
                               (const void*)write_kernel<WC_SCHEME_DITHER_INT8, 10, true, 1>,
                               (const void*)write_kernel<WC_SCHEME_DITHER_INT8, 10, true, 2>,
                               (const void*)write_kernel<WC_SCHEME_DITHER_INT8_G32, 8, true, 1>,
                               (const void*)write_kernel<WC_SCHEME_DITHER_INT8_G32, 8, true, 2>};
        for (const void* f : fns) {
            cudaError_t e = cudaFuncSetAttribute(f, cudaFuncAttributePreferredSharedMemoryCarveout,
                                                 (int)cudaSharedmemCarveoutMaxShared);
            if (e != cudaSuccess) return e;
        }
        return cudaSuccess;
    });
    if (set != cudaSuccess) return set;
    const bool per_head = p.n_tok >= kPerHeadMinTokens;
    const bool two = write_two_tasks(scheme, bits, p.n_tok, p.num_kv_heads);
    const int upc = write_units_per_cta(two ? 2 : 1);
    const dim3 grid = per_head ? dim3((p.n_tok + upc - 1) / upc, p.num_kv_heads)
                               : dim3((p.n_tok * p.num_kv_heads + upc - 1) / upc);
    auto go = [&](auto kernel) { return launch_pdl(kernel, grid, dim3(128), 0, stream, p); };
    if (scheme == WC_SCHEME_FP8_E4M3)
        return two ? go(write_kernel<WC_SCHEME_FP8_E4M3, 8, true, 2>) : go(write_kernel<WC_SCHEME_FP8_E4M3, 8, false, 1>);
    if (scheme == WC_SCHEME_DITHER_INT8_G32)
        return two        ? go(write_kernel<WC_SCHEME_DITHER_INT8_G32, 8, true, 2>)
               : per_head ? go(write_kernel<WC_SCHEME_DITHER_INT8_G32, 8, true, 1>)
                          : go(write_kernel<WC_SCHEME_DITHER_INT8_G32, 8, false, 1>);
    if (bits == 8)
        return two ? go(write_kernel<WC_SCHEME_DITHER_INT8, 8, true, 2>)
                   : go(write_kernel<WC_SCHEME_DITHER_INT8, 8, false, 1>);
    return two        ? go(write_kernel<WC_SCHEME_DITHER_INT8, 10, true, 2>)
           : per_head ? go(write_kernel<WC_SCHEME_DITHER_INT8, 10, true, 1>)
                      : go(write_kernel<WC_SCHEME_DITHER_INT8, 10, false, 1>);
}

}  // namespace wc
