// vie_recall.cu - Recall@k bookkeeping on the device (paper, Section 4.3:
// recall is the share of the exact head's top-k tokens that an approximate
// search also retrieves, over many hidden states).
//
// Per query q: hits[q] = #{ j < k : exact[q, j] >= 0 and exact[q, j] is among
// approx[q, 0..m-1] }.  The candidates act as a set (a repeated candidate is
// found once per exact entry) and negative entries are empty slots.  Integer
// work only: the result is exact.
//
// Bound: reading the lists, 4 n (k + m) bytes (6.5 us at n = 20000, k = 50,
// m = 500).  Comparing every candidate with every exact entry costs k m
// operations per query instead (212 us there, 24.9 us as below); so
//   k <= 8   every lane keeps all k exact entries in registers and compares
//            its own candidates with them (a bit per entry, OR-ed over the
//            warp at the end);
//   k > 8 and m <= 32
//            the other way round: every lane keeps all m candidates and
//            compares its own exact entries with them (a table would be built
//            for a few look-ups: n = 20000, k = 1000: 15 us at m = 1 instead
//            of 90, 43 at m = 32 instead of 95);
//   else     the exact entries go into a hash table in shared memory (open
//            addressing, at most a quarter full), each with the number of
//            positions that hold it; a candidate that finds its entry takes
//            that number and leaves 0, so a repeat adds nothing.  Most
//            candidates are no hits, and a warp runs as long as its longest
//            probe, so a bit map of the entries' hashes (8 bits per slot, at
//            most 3 % set) is tested first, eight candidates per lane without
//            a branch, and only the survivors probe.
#include <cuda_runtime.h>

#include <cstdint>

#include "vie_device.cuh"
#include "vie_launch.h"

namespace vie {

constexpr int kRecallWarps = 8;
constexpr int kRecallUnroll = 8;  // candidates in flight per lane

// k <= K: one warp per query, candidates lane, lane + 32, ...
template <int K>
__global__ void __launch_bounds__(kRecallWarps * 32) recall_direct_kernel(const int32_t *__restrict__ exact,
                                                                         int k,
                                                                         const int32_t *__restrict__ approx,
                                                                         int m, int64_t n,
                                                                         int32_t *__restrict__ hits) {
    griddep_wait();  // the lists may come from the kernels before this one
    const int lane = threadIdx.x & 31;
    const int64_t q = static_cast<int64_t>(blockIdx.x) * kRecallWarps + (threadIdx.x >> 5);
    if (q >= n) return;
    int32_t e[K];
#pragma unroll
    for (int j = 0; j < K; ++j) e[j] = j < k ? exact[q * k + j] : -1;
    uint32_t found = 0;
    const int32_t *aq = approx + q * m;
    for (int i0 = lane; i0 < m; i0 += 32 * kRecallUnroll) {
        int32_t a[kRecallUnroll];
#pragma unroll
        for (int u = 0; u < kRecallUnroll; ++u) a[u] = i0 + 32 * u < m ? aq[i0 + 32 * u] : -1;
#pragma unroll
        for (int u = 0; u < kRecallUnroll; ++u)
#pragma unroll
            for (int j = 0; j < K; ++j) found |= static_cast<uint32_t>(a[u] == e[j]) << j;
    }
#pragma unroll
    for (int j = 0; j < K; ++j)  // an empty exact entry is never a hit
        if (e[j] < 0) found &= ~(1u << j);
    found = __reduce_or_sync(0xFFFFFFFFu, found);
    if (lane == 0) hits[q] = __popc(found);
}

// m <= M: one warp per query, exact entries lane, lane + 32, ..., U at a time.
template <int M, int U>
__global__ void __launch_bounds__(kRecallWarps * 32) recall_few_kernel(const int32_t *__restrict__ exact, int k,
                                                                      const int32_t *__restrict__ approx, int m,
                                                                      int64_t n, int32_t *__restrict__ hits) {
    griddep_wait();  // the lists may come from the kernels before this one
    const int lane = threadIdx.x & 31;
    const int64_t q = static_cast<int64_t>(blockIdx.x) * kRecallWarps + (threadIdx.x >> 5);
    if (q >= n) return;
    const int32_t *eq = exact + q * k;
    int32_t a[M];
#pragma unroll
    for (int j = 0; j < M; ++j) a[j] = j < m ? approx[q * m + j] : -1;
    unsigned sum = 0;
    for (int i0 = lane; i0 < k; i0 += 32 * U) {
        int32_t e[U];
#pragma unroll
        for (int u = 0; u < U; ++u) e[u] = i0 + 32 * u < k ? eq[i0 + 32 * u] : -1;
#pragma unroll
        for (int u = 0; u < U; ++u) {
            bool in = false;
#pragma unroll
            for (int j = 0; j < M; ++j) in |= e[u] == a[j];
            sum += in && e[u] >= 0 ? 1u : 0u;  // an empty exact entry is never a hit
        }
    }
    sum = __reduce_add_sync(0xFFFFFFFFu, sum);
    if (lane == 0) hits[q] = static_cast<int32_t>(sum);
}

// k > 8: WPQ warps per query (1, or all kRecallWarps of the CTA), a table of
// 1 << log2_slots >= 4 k slots per query: its keys, its counts, its bit map.
template <int WPQ>
__global__ void __launch_bounds__(kRecallWarps * 32) recall_hash_kernel(const int32_t *__restrict__ exact,
                                                                       int k,
                                                                       const int32_t *__restrict__ approx,
                                                                       int m, int64_t n, int log2_slots,
                                                                       int32_t *__restrict__ hits) {
    extern __shared__ __align__(16) unsigned char recall_smem[];
    __shared__ int part[kRecallWarps];
    constexpr int kPerCta = kRecallWarps / WPQ;  // queries per CTA
    constexpr int T = 32 * WPQ;                  // threads of a query
    const int lane = threadIdx.x & 31, warp = threadIdx.x >> 5;
    const int t = WPQ == 1 ? lane : static_cast<int>(threadIdx.x);
    const int slots = 1 << log2_slots, mask = slots - 1, shift = 32 - log2_slots;
    int32_t *key = reinterpret_cast<int32_t *>(recall_smem + (WPQ == 1 ? warp : 0) * 9 * slots);
    int32_t *cnt = key + slots;
    uint32_t *bits = reinterpret_cast<uint32_t *>(cnt + slots);  // 8 per slot
    auto sync = [] {
        if constexpr (WPQ == 1) __syncwarp();
        else __syncthreads();
    };
    // an empty table: keys -1, counts and bits 0 (overlaps the kernel before this one)
    int4 *key4 = reinterpret_cast<int4 *>(key);
    for (int i = t; i < slots / 4; i += T) key4[i] = make_int4(-1, -1, -1, -1);
    for (int i = slots / 4 + t; i < slots / 2 + slots / 16; i += T) key4[i] = make_int4(0, 0, 0, 0);
    sync();
    griddep_wait();  // the lists may come from the kernels before this one
    const int64_t q = static_cast<int64_t>(blockIdx.x) * kPerCta + (WPQ == 1 ? warp : 0);
    if (q >= n) return;  // whole warps (WPQ = 1), never part of a CTA (one query per CTA)
    const int32_t *eq = exact + q * k, *aq = approx + q * m;
    auto hash = [](int32_t v) { return static_cast<uint32_t>(v) * 0x9E3779B1u; };
    for (int j = t; j < k; j += T) {
        const int32_t v = eq[j];
        if (v < 0) continue;
        const uint32_t hv = hash(v), bit = hv >> (shift - 3);
        atomicOr(&bits[bit >> 5], 1u << (bit & 31));
        for (int s = static_cast<int>(hv >> shift);; s = (s + 1) & mask) {  // ends: the table is never full
            const int32_t old = atomicCAS(&key[s], -1, v);
            if (old == -1 || old == v) {
                atomicAdd(&cnt[s], 1);
                break;
            }
        }
    }
    sync();
    int sum = 0;
    for (int i0 = t; i0 < m; i0 += T * kRecallUnroll) {
        int32_t a[kRecallUnroll];
        uint32_t left = 0;  // candidates that may be entries
#pragma unroll
        for (int u = 0; u < kRecallUnroll; ++u) a[u] = i0 + T * u < m ? aq[i0 + T * u] : -1;
#pragma unroll
        for (int u = 0; u < kRecallUnroll; ++u) {
            const uint32_t bit = hash(a[u]) >> (shift - 3);
            const uint32_t set = (bits[bit >> 5] >> (bit & 31)) & 1u;
            left |= (a[u] >= 0 ? set : 0u) << u;
        }
        // one probe step of one candidate per turn, the next candidate (read
        // again, from L1) as soon as the last is settled
        int32_t v = -1;
        int s = 0;
        while (true) {
            if (v < 0) {
                if (left == 0) break;
                v = aq[i0 + T * (__ffs(left) - 1)];
                left &= left - 1;
                s = static_cast<int>(hash(v) >> shift);
            }
            const int32_t x = key[s];
            if (x == v) sum += atomicExch(&cnt[s], 0);
            if (x == v || x == -1) v = -1;
            s = (s + 1) & mask;
        }
    }
    __syncwarp();
    sum = static_cast<int>(__reduce_add_sync(0xFFFFFFFFu, static_cast<unsigned>(sum)));
    if constexpr (WPQ == 1) {
        if (lane == 0) hits[q] = sum;
    } else {
        if (lane == 0) part[warp] = sum;
        __syncthreads();
        if (threadIdx.x == 0) {
            int total = 0;
#pragma unroll
            for (int w = 0; w < kRecallWarps; ++w) total += part[w];
            hits[q] = total;
        }
    }
}

cudaError_t launch_recall_hits(const int32_t *exact, int k, const int32_t *approx, int m, int64_t n,
                               int32_t *hits, cudaStream_t stream) {
    cudaLaunchConfig_t cfg = {};
    cfg.gridDim = dim3(static_cast<unsigned>((n + kRecallWarps - 1) / kRecallWarps));
    cfg.blockDim = dim3(kRecallWarps * 32);
    cfg.stream = stream;
    cudaLaunchAttribute attr[1];
    attr[0].id = cudaLaunchAttributeProgrammaticStreamSerialization;
    attr[0].val.programmaticStreamSerializationAllowed = 1;
    cfg.attrs = attr;
    cfg.numAttrs = 1;
    if (k <= 2) return cudaLaunchKernelEx(&cfg, recall_direct_kernel<2>, exact, k, approx, m, n, hits);
    if (k <= 8) return cudaLaunchKernelEx(&cfg, recall_direct_kernel<8>, exact, k, approx, m, n, hits);
    if (m <= 32) {
        const auto few = m <= 8 ? (k <= 128 ? recall_few_kernel<8, 4> : recall_few_kernel<8, 8>)
                                : (m <= 16 ? (k <= 128 ? recall_few_kernel<16, 4> : recall_few_kernel<16, 8>)
                                           : (k <= 128 ? recall_few_kernel<32, 4> : recall_few_kernel<32, 8>));
        return cudaLaunchKernelEx(&cfg, few, exact, k, approx, m, n, hits);
    }
    int log2_slots = 6;
    while ((1 << log2_slots) < 4 * k) ++log2_slots;
    const size_t table = size_t(9) << log2_slots;
    // A warp per query while its table is small (at most 4.5 KB, so the CTAs'
    // tables do not limit the warps in flight) and the queries fill the
    // chip; otherwise the eight warps of a CTA share one query's table and
    // split its candidates.
    const bool cta_per_query = log2_slots > 9 || (n < 4096 && m >= 1024);
    if (cta_per_query) {
        cfg.gridDim = dim3(static_cast<unsigned>(n));
        cfg.dynamicSmemBytes = table;
        return cudaLaunchKernelEx(&cfg, recall_hash_kernel<kRecallWarps>, exact, k, approx, m, n, log2_slots, hits);
    }
    cfg.dynamicSmemBytes = table * kRecallWarps;
    return cudaLaunchKernelEx(&cfg, recall_hash_kernel<1>, exact, k, approx, m, n, log2_slots, hits);
}

}  // namespace vie
