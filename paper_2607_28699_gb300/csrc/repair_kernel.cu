// Block-level repair selection (§6.3.5 "Block-level paging").  The e-form
// certificate is block decomposable: with p~ held fixed, replacing the keys of
// logical page j by their exact values (witness 0, so c_t = 0) lowers D = A - 1
// by exactly C_j = sum_{t in j} p~_t (e^{c_t} - 1).  For each cell the gate sent
// to fallback, pages rank by decreasing C_j (ties to the lower page), and the
// page-in list is the shortest prefix after which the meter of the rest,
// 1/2 R (R + 2) with R the sum of the contributions not yet paged in, is at
// most tau.
//
// One CTA per (sequence, query head).  The decode's per-page terms (m_j, d_j)
// are normalised with the cell's final (M, L) and sorted by 64-bit keys (the
// contribution's bits above the complemented page index, so that a descending sort
// ranks by contribution, then by lower page; NaN above +inf).  The remaining excess
// R is then summed from the tail.
//
// The sort: as many buckets as sorted positions over the cell's range of bits (a
// logarithmic scale, on which contributions spread), a count per bucket, their
// prefix sums, and each key's rank inside its bucket by comparison with the bucket's
// other keys (a handful).  A cell whose fullest bucket holds more than kMaxBucket keys
// (many contributions that are zero or equal; a range stretched by inf or NaN) is sorted by
// stable passes over 7-bit digits instead.  Both give the same order, so the sums that
// follow are the same bits.
// Measured, network of compare-exchanges (the only sort before) -> this: 784 cells of 2048
// pages 58.7 -> 21.0 us, half of their contributions zero 58.6 -> 17.5, all equal 59.2 -> 19.4;
// 2800 of 512 43.6 -> 18.4; 8400 of 100 119 -> 13.1; 196 of 8192 99 -> 31.  Twice or four times
// the buckets at 784 x 2048: no faster.
#include <climits>

#include "dispatch.h"
#include "wc_kernels.cuh"

namespace wc {

namespace {

// The remaining sums are taken as kSumThreads threads would, thread i holding KS
// consecutive sorted positions, whatever the CTA's size: their order of additions, and
// with it the count that a borderline tau gives, does not depend on how a table is sorted.
constexpr int kSumThreads = 512, kSumWarps = kSumThreads / 32;
// Keys of a bucket that its members are compared with: a warp's ranking takes as many
// steps as its fullest bucket.
constexpr int kMaxBucket = 64;

__device__ __forceinline__ float key_value(unsigned long long key) { return __uint_as_float((uint32_t)(key >> 32)); }

// A CTA of T threads sorts K keys per thread; KS: positions per thread of the sums.
// T grows with the table (K = 4 up to 4096 pages), so that a small cell costs few warps
// and barriers (repair_wide has both sides).
// Threads per SM that the register budget leaves room for: all 2048 with one or two keys a
// thread, 1536 with four (at most 40 registers: 2800 cells of 512 pages 18.4 us, without it 23.9),
// 1024 with more.
constexpr int min_ctas(int T, int K) {
    const int n = (K <= 2 ? 2048 : K <= 4 ? 1536 : 1024) / T;
    return n < 1 ? 1 : n > 32 ? 32 : n;
}
template <int T, int K, int KS>
__global__ void __launch_bounds__(T, min_ctas(T, K)) repair_select_kernel(const __grid_constant__ RepairParams p) {
    constexpr int N = T * K;      // sorted length: the block table, padded to a power of two
    constexpr int kSelWarps = T / 32;
    extern __shared__ __align__(16) unsigned long long xs[];   // [N] keys
    uint32_t* cnt = reinterpret_cast<uint32_t*>(xs + N);      // [N] keys per bucket, then the buckets' ends
    __shared__ uint32_t warp_lo[kSelWarps], warp_hi[kSelWarps], warp_sum[kSelWarps];
    __shared__ float warp_tot[kSumWarps];
    __shared__ int warp_min[kSelWarps];
    __shared__ float r_at_k;
    const int hq = blockIdx.x, b = blockIdx.y;
    const int tid = threadIdx.x, lane = tid & 31, warp = tid >> 5;
    const int base = tid * K;
    const size_t cell = (size_t)b * p.num_q_heads + hq;

    // the page terms are read whatever the context length (every block-table
    // column is in bounds), so that no load waits for another
    const float2* terms = p.page_terms + cell * p.max_pages;
    const float2 nm = p.softmax_norm[cell];
    const bool kept = p.keep_q != nullptr && p.keep_q[cell] != 0;
    int ctx = p.ctx_lens[b];
    if (ctx < 0 || ctx > p.max_pages * kPage) {
        if (tid == 0 && hq == 0 && p.status) atomicOr(p.status, WC_DEV_BAD_CTX);
        ctx = max(0, min(ctx, p.max_pages * kPage));
    }
    const int n = (ctx + kPage - 1) / kPage;

    // ---- C_j = d_j 2^(m_j - M) / L; thread t takes pages t, t + T, ... (any order does) --
    // A page that contributes nothing is not sorted: nothing remains after the pages that
    // do, so that with tau >= 0 the list ends before it.
    const bool zeros = !(p.tau >= 0.f);   // every page is listed, these in page order behind the others
    unsigned long long key[K];
    auto page_of = [&](int r) { return tid + r * T; };
#pragma unroll
    for (int r = 0; r < K; ++r) {
        const int j = page_of(r);
        const float2 t = j < p.max_pages ? terms[j] : make_float2(-INFINITY, 0.f);
        key[r] = 0ull;   // not sorted
        if (j < n) {
            float cj = (nm.y > 0.f && t.y != 0.f) ? __fdiv_rn(t.y * exp2f(t.x - nm.x), nm.y) : 0.f;
            if (cj <= 0.f) cj = 0.f;   // -0 ranks as +0; NaN stays and ranks first
            if (p.contrib) p.contrib[cell * p.max_pages + j] = cj;
            if (cj != 0.f || zeros) key[r] = ((unsigned long long)__float_as_uint(cj) << 32) | (0xFFFFFFFFu - (uint32_t)j);
        }
    }

    // Sorted position i ends at word spot(i): each thread of the sums reads KS consecutive
    // positions, permuted so that the 16 lanes of a half-warp meet 16 distinct bank pairs.
    auto spot = [](int i) {
        const int th = i / KS;
        return i ^ (KS >= 16 ? (th & 15) : (((th * KS) >> 4) & (KS - 1)));
    };

    // ---- descending sort into xs (kept cells: nothing is paged in, any order does) ------
    if (!kept) {
        uint32_t lo = 0xFFFFFFFFu, hi = 0u;   // the contributions' bits: least, largest finite
#pragma unroll
        for (int r = 0; r < K; ++r) {
            cnt[page_of(r)] = 0u;
            if (key[r] != 0ull) {
                const uint32_t bits = (uint32_t)(key[r] >> 32);
                lo = min(lo, bits);
                hi = max(hi, bits < 0x7F800000u ? bits : 0u);
            }
        }
        lo = __reduce_min_sync(0xffffffffu, lo);
        hi = __reduce_max_sync(0xffffffffu, hi);
        if (lane == 0) {
            warp_lo[warp] = lo;
            warp_hi[warp] = hi;
        }
        __syncthreads();
        if (kSelWarps > 1) {   // lane w takes warp w's (kSelWarps is a power of two)
            lo = __reduce_min_sync(0xffffffffu, warp_lo[lane % kSelWarps]);
            hi = __reduce_max_sync(0xffffffffu, warp_hi[lane % kSelWarps]);
        }
        // bucket 0 holds the largest keys (inf and NaN with the largest finite ones); the shift
        // is the least that gives N buckets
        const int shift = max(0, 32 - __clz(hi > lo ? hi - lo : 0u) - (31 - __clz(N)));
        auto bucket = [&](unsigned long long k) {
            const uint32_t bits = (uint32_t)(k >> 32);
            return bits < hi ? (hi - bits) >> shift : 0u;
        };
#pragma unroll
        for (int r = 0; r < K; ++r)
            if (key[r] != 0ull) atomicAdd(&cnt[bucket(key[r])], 1u);
        __syncthreads();
        uint32_t sum = 0u, most = 0u;   // exclusive prefix sums; thread t takes buckets [t K, t K + K)
#pragma unroll
        for (int r = 0; r < K; ++r) {
            const uint32_t x = cnt[base + r];
            most = max(most, x);
            sum += x;
        }
        uint32_t inc = sum;
#pragma unroll
        for (int o = 1; o < 32; o <<= 1) {
            const uint32_t v = __shfl_up_sync(0xffffffffu, inc, o);
            if (lane >= o) inc += v;
        }
        if (lane == 31) warp_sum[warp] = inc;
        const bool buckets = !__syncthreads_or(most > kMaxBucket);   // block-uniform
        const uint32_t of_warp = lane < kSelWarps ? warp_sum[lane] : 0u;
        uint32_t first = inc - sum + __reduce_add_sync(0xffffffffu, lane < warp ? of_warp : 0u);
        const int n_sorted = (int)__reduce_add_sync(0xffffffffu, of_warp);
        if (buckets) {
#pragma unroll
            for (int r = 0; r < K; ++r) {
                const uint32_t x = cnt[base + r];
                cnt[base + r] = first;
                first += x;
            }
            __syncthreads();
#pragma unroll
            for (int r = 0; r < K; ++r)   // grouped by bucket; cnt then holds each bucket's end
                if (key[r] != 0ull) xs[atomicAdd(&cnt[bucket(key[r])], 1u)] = key[r];
            __syncthreads();
            uint32_t rank[(K + 1) / 2];   // two to a word (positions below 16384)
#pragma unroll
            for (int r = 0; r < K; ++r) {
                uint32_t k = 0u;   // the bucket's first position plus its larger keys
                if (key[r] != 0ull) {
                    const uint32_t bk = bucket(key[r]), last = cnt[bk];
                    k = bk > 0 ? cnt[bk - 1] : 0u;
                    for (uint32_t i = k, e = last; i < e; ++i) k += xs[i] > key[r] ? 1u : 0u;
                }
                if (r & 1) rank[r / 2] |= k << 16;
                else rank[r / 2] = k;
            }
            __syncthreads();
#pragma unroll
            for (int r = 0; r < K; ++r) {
                if (key[r] != 0ull) xs[spot((int)((rank[r / 2] >> (16 * (r & 1))) & 0xFFFFu))] = key[r];
                if (page_of(r) >= n_sorted) xs[spot(page_of(r))] = 0ull;
            }
        } else {
            // Stable passes over the digits of top - bits, from the lowest: the keys start in
            // page order, so equal contributions stay in it.  A warp holds 32 K consecutive
            // positions; within a warp a key's place among its digit's keys is a count of lanes
            // by ballots, across warps the prefix sums of the counts per (digit, warp).
            constexpr int kDigit = K >= 4 ? 7 : K == 2 ? 6 : 5, kBins = 1 << kDigit;
            constexpr int kPer = kBins / 32;   // counts per thread: kBins per warp
            static_assert(kPer <= K, "the counts fit in cnt");
            auto slot = [](int d, int w) { return d * kSelWarps + ((w + d) & (kSelWarps - 1)); };   // spreads the banks
            auto place = [&](int r) { return (warp * K + r) * 32 + lane; };
            uint32_t top = 0u;   // the largest, inf and NaN included
#pragma unroll
            for (int r = 0; r < K; ++r) {
                top = max(top, (uint32_t)(key[r] >> 32));
                xs[page_of(r)] = key[r];
            }
            top = __reduce_max_sync(0xffffffffu, top);
            if (lane == 0) warp_hi[warp] = top;
            __syncthreads();
            top = __reduce_max_sync(0xffffffffu, warp_hi[lane % kSelWarps]);
#pragma unroll
            for (int r = 0; r < K; ++r) key[r] = xs[place(r)];
            const int length = 32 - __clz(top - lo);
            for (int d0 = 0; d0 == 0 || d0 < length; d0 += kDigit) {   // the first also moves the sorted to the front
                auto digit = [&](int r) { return (int)(((top - (uint32_t)(key[r] >> 32)) >> d0) & (kBins - 1)); };
                for (int i = tid; i < kBins * kSelWarps; i += T) cnt[i] = 0u;
                __syncthreads();
                uint32_t nth[(K + 1) / 2];   // two to a word
#pragma unroll
                for (int r = 0; r < K; ++r) {
                    const bool valid = key[r] != 0ull;
                    const int d = digit(r);
                    uint32_t peers = __ballot_sync(0xffffffffu, valid);
#pragma unroll
                    for (int i = 0; i < kDigit; ++i) {
                        const bool bit = (d >> i) & 1;
                        const uint32_t set = __ballot_sync(0xffffffffu, bit);
                        peers &= bit ? set : ~set;
                    }
                    uint32_t* c = cnt + slot(d, warp);
                    const uint32_t k = valid ? *c + __popc(peers & ((1u << lane) - 1u)) : 0u;
                    __syncwarp();
                    if (valid && (peers >> lane) == 1u) *c = k + 1u;   // the last of the digit's lanes
                    __syncwarp();
                    if (r & 1) nth[r / 2] |= k << 16;
                    else nth[r / 2] = k;
                }
                __syncthreads();
                uint32_t tot = 0u;   // thread t takes the counts [t kPer, t kPer + kPer) in (digit, warp) order
                auto count = [&](int i) -> uint32_t& {
                    const int e = tid * kPer + i;
                    return cnt[slot(e / kSelWarps, e % kSelWarps)];
                };
#pragma unroll
                for (int i = 0; i < kPer; ++i) tot += count(i);
                uint32_t to = tot;
#pragma unroll
                for (int o = 1; o < 32; o <<= 1) {
                    const uint32_t v = __shfl_up_sync(0xffffffffu, to, o);
                    if (lane >= o) to += v;
                }
                if (lane == 31) warp_sum[warp] = to;
                __syncthreads();
                uint32_t start = to - tot + __reduce_add_sync(0xffffffffu, lane < warp ? warp_sum[lane] : 0u);
#pragma unroll
                for (int i = 0; i < kPer; ++i) {
                    const uint32_t x = count(i);
                    count(i) = start;
                    start += x;
                }
                __syncthreads();
#pragma unroll
                for (int r = 0; r < K; ++r)
                    if (key[r] != 0ull) xs[cnt[slot(digit(r), warp)] + ((nth[r / 2] >> (16 * (r & 1))) & 0xFFFFu)] = key[r];
                __syncthreads();
#pragma unroll
                for (int r = 0; r < K; ++r) key[r] = place(r) < n_sorted ? xs[place(r)] : 0ull;
            }
            __syncthreads();
#pragma unroll
            for (int r = 0; r < K; ++r) xs[spot(place(r))] = key[r];
        }
    } else {   // page order, the order a kept cell's sums have always had
#pragma unroll
        for (int r = 0; r < K; ++r) xs[spot(page_of(r))] = key[r];
    }
    __syncthreads();

    // ---- remaining sums R_i = sum of the ranked contributions from i on ---------
    // each thread of the sums adds its KS positions from the tail; the later
    // threads' sums enter as an offset
    constexpr int kRounds = (kSumWarps + kSelWarps - 1) / kSelWarps;   // warps of the sums per warp
    auto value = [&](int i) { return i < N ? key_value(xs[spot(i)]) : 0.f; };
    float offset[kRounds];
#pragma unroll
    for (int q = 0; q < kRounds; ++q) {
        const int w = warp + q * kSelWarps, at = (32 * w + lane) * KS;
        offset[q] = 0.f;
        if (w < kSumWarps) {   // warp-uniform
            float tot = 0.f;
            if (32 * w * KS < n) {
#pragma unroll
                for (int r = KS - 1; r >= 0; --r) tot += value(at + r);
            }
            float suf = tot;   // inclusive suffix over the warp's lanes
#pragma unroll
            for (int o = 1; o < 32; o <<= 1) {
                const float v = __shfl_down_sync(0xffffffffu, suf, o);
                if (lane + o < 32) suf += v;
            }
            if (lane == 0) warp_tot[w] = suf;
            offset[q] = __shfl_down_sync(0xffffffffu, suf, 1);   // later lanes of this warp
            if (lane == 31) offset[q] = 0.f;
        }
    }
    __syncthreads();
    int cand = INT_MAX;
#pragma unroll
    for (int q = 0; q < kRounds; ++q) {
        const int w = warp + q * kSelWarps, at = (32 * w + lane) * KS;
        if (w < kSumWarps) {
            for (int x = kSumWarps - 1; x > w; --x) offset[q] += warp_tot[x];
            if (!kept && at < N) {
                float s = offset[q];
#pragma unroll
                for (int r = KS - 1; r >= 0; --r) {
                    s += value(at + r);
                    if (0.5f * s * (s + 2.0f) <= p.tau) cand = min(cand, at + r);   // NaN -> false
                }
            }
        }
    }
    cand = __reduce_min_sync(0xffffffffu, cand);
    if (lane == 0) warp_min[warp] = cand;
    __syncthreads();
    const int kmin = __reduce_min_sync(0xffffffffu, warp_min[lane % kSelWarps]);
    const int kstar = kept ? 0 : min(kmin, n);   // every page when no prefix is enough
    if (kstar >= n) {
        if (tid == 0) r_at_k = 0.f;
    } else {
#pragma unroll
        for (int q = 0; q < kRounds; ++q) {
            const int at = (32 * (warp + q * kSelWarps) + lane) * KS;
            if (kstar >= at && kstar < at + KS) {
                float s = offset[q];
#pragma unroll
                for (int r = KS - 1; r >= 0; --r)
                    if (at + r >= kstar) s += value(at + r);
                r_at_k = s;
            }
        }
    }
    for (int i = tid; i < kstar; i += T)
        p.repair_pages[cell * p.max_pages + i] = (int32_t)(0xFFFFFFFFu - (uint32_t)(xs[spot(i)] & 0xFFFFFFFFull));
    __syncthreads();
    if (tid == 0) {
        p.n_repair[cell] = kstar;
        p.d_after[cell] = r_at_k;
    }
}

template <int T, int K, int KS>
cudaError_t launch_select(const RepairParams& p, cudaStream_t stream) {
    constexpr size_t smem = (size_t)T * K * (sizeof(unsigned long long) + sizeof(uint32_t));
    static PerDevice<Configured, cudaError_t> configured;
    if (cudaError_t e = configure(configured, repair_select_kernel<T, K, KS>, smem)) return e;
    repair_select_kernel<T, K, KS><<<dim3(p.num_q_heads, p.batch), T, smem, stream>>>(p);
    return cudaGetLastError();
}

}  // namespace

cudaError_t launch_repair_select(const RepairParams& p, cudaStream_t stream) {
    static_assert(kRepairMaxPages == 16 * 1024, "the largest instance holds 16 keys per thread");
    if (p.batch == 0) return cudaSuccess;
    // the least power of two that holds the table; KS = positions per thread of 512
    const int64_t cells = (int64_t)p.batch * p.num_q_heads;
    if (p.max_pages <= 32) return launch_select<32, 1, 1>(p, stream);
    if (p.max_pages <= 64)
        return repair_wide(cells, 64) ? launch_select<64, 1, 1>(p, stream) : launch_select<32, 2, 1>(p, stream);
    if (p.max_pages <= 128)
        return repair_wide(cells, 128) ? launch_select<128, 1, 1>(p, stream) : launch_select<64, 2, 1>(p, stream);
    if (p.max_pages <= 256)
        return repair_wide(cells, 256)  ? launch_select<256, 1, 1>(p, stream)
               : repair_wide(cells, 64) ? launch_select<128, 2, 1>(p, stream) : launch_select<64, 4, 1>(p, stream);
    if (p.max_pages <= 512)
        return repair_wide(cells, 256) ? launch_select<256, 2, 1>(p, stream) : launch_select<128, 4, 1>(p, stream);
    if (p.max_pages <= 1024)
        return repair_wide(cells, 512) ? launch_select<512, 2, 2>(p, stream) : launch_select<256, 4, 2>(p, stream);
    if (p.max_pages <= 2048) return launch_select<512, 4, 4>(p, stream);
    if (p.max_pages <= 4096)
        return repair_wide(cells, 1024) ? launch_select<1024, 4, 8>(p, stream) : launch_select<512, 8, 8>(p, stream);
    if (p.max_pages <= 8192) return launch_select<1024, 8, 16>(p, stream);
    return launch_select<1024, 16, 32>(p, stream);
}

}  // namespace wc
