// vie_tc_many.cu - the filtered GEMM for many queries (vie_tc_many.cuh), the
// bounds from its sample, the final top-k of each query's candidates, and
// their launchers.
#include "vie_launch.h"
#include "vie_stream_topk.cuh"
#include "vie_tc_launch.cuh"
#include "vie_tc_many.cuh"
#include "vie_tcgen05.cuh"

namespace vie {

struct MnMisc {
    uint32_t tmem_base;
    int abort;
};

__global__ void __cluster_dims__(2, 1, 1) __launch_bounds__(kMnThreads, 1)
    tc_many_kernel(const __grid_constant__ CUtensorMap mapW, const __grid_constant__ CUtensorMap mapH,
                   const MnParams p) {
    extern __shared__ __align__(1024) unsigned char mn_smem[];
    uint64_t *full = reinterpret_cast<uint64_t *>(mn_smem);
    uint64_t *empty = full + kMnStages;
    uint64_t *tfull = empty + kMnStages;
    uint64_t *tempty = tfull + 2;
    uint64_t *final_bar = tempty + 2;
    MnMisc *mc = reinterpret_cast<MnMisc *>(mn_smem + 512);
    unsigned char *ring = mn_smem + 1024;
    ring += (1024u - (smem_addr(ring) & 1023u)) & 1023u;
    volatile int *abort_flag = &mc->abort;

    const int tid = threadIdx.x, warp = tid >> 5, lane = tid & 31;
    const uint32_t rank = cluster_ctarank();
    const int pair = blockIdx.x >> 1, n_pairs = gridDim.x >> 1;
    const int n_kb = (p.d_pad + 63) / 64;
    const int n_items = static_cast<int>((p.rows + kMnRows - 1) / kMnRows) * p.groups;

    if (tid == 0) {
        for (int s = 0; s < kMnStages; ++s) {
            mbar_init(&full[s], 1);
            mbar_init(&empty[s], 1);
        }
        for (int b = 0; b < 2; ++b) {
            mbar_init(&tfull[b], 1);
            mbar_init(&tempty[b], 2 * kMnEpiWarps);
        }
        mbar_init(final_bar, 1);
        mc->abort = 0;
        fence_mbar_init();
    }
    if (warp == 1) {
        tmem_alloc_pair(&mc->tmem_base, 512);
        tmem_relinquish_pair();
        tc_fence_before_sync();
    }
    __syncthreads();
    cluster_sync();  // the pair's barriers are set up before either CTA signals the other's
    tc_fence_after_sync();
    const uint32_t tmem = mc->tmem_base;
    if (tid == 0) griddep_launch_dependents();

    // Items in order: the groups of one tile of W are neighbours, so that the
    // pairs that run them together read the tile from HBM once.
    if (warp == 0) {
        // ---------------- TMA producer ----------------
        if (lane == 0) {
            tma_prefetch_map(&mapW);
            tma_prefetch_map(&mapH);
            griddep_wait();  // the query matrix comes from the kernel before this one
            int it = 0, issued = 0;
            bool ok = true;
            for (int item = pair; item < n_items && ok; item += n_pairs) {
                const int tile = item / p.groups, g = item - tile * p.groups;
                for (int kb = 0; kb < n_kb; ++kb, ++it) {
                    const int s = it % kMnStages, u = it / kMnStages;
                    if (it >= kMnStages && !mbar_wait(&empty[s], (u - 1) & 1, abort_flag)) {
                        ok = false;
                        break;
                    }
                    unsigned char *st = ring + s * kMnStageBytes;
                    if (rank == 0) mbar_arrive_expect_tx(&full[s], 2 * kMnStageBytes);
                    const uint32_t bar = cluster_map(&full[s], 0);
                    tma_load_2d_pair(st, &mapW, kb * 64, tile * kMnRows + static_cast<int>(rank) * 128, bar);
                    tma_load_2d_pair(st + kMnStageBytes / 2, &mapH, kb * 64,
                                     g * 2 * kMnGroup + static_cast<int>(rank) * 128, bar);
                    issued = it + 1;
                }
            }
            if (!ok) {
                atomicOr(p.err, kErrWaitTimeout);
                mc->abort = 1;
                // copies in flight land before the CTA exits: the leader can
                // watch its barriers, the other CTA gives them a millisecond
                const int never = 0;
                if (rank == 0)
                    for (int t2 = max(0, issued - kMnStages); t2 < issued; ++t2)
                        mbar_wait(&full[t2 % kMnStages], (t2 / kMnStages) & 1, const_cast<volatile int *>(&never));
                const uint64_t t0 = global_timer_ns();
                while (global_timer_ns() - t0 < 1000000ull) {
                }
            }
        }
        __syncwarp();
    } else if (warp == 1) {
        // ---------------- MMA issuer (the leader's) ----------------
        if (lane == 0 && rank == 0) {
            griddep_wait();  // the limit of the waits below counts from here, not from a start under an earlier kernel
            constexpr uint32_t idesc = umma_idesc_bf16_f32(kMnRows, 2 * kMnGroup);
            int it = 0, ti = 0;
            bool ok = true;
            for (int item = pair; item < n_items && ok; item += n_pairs, ++ti) {
                const int b = ti & 1, ub = ti >> 1;
                if (ti >= 2 && !mbar_wait(&tempty[b], (ub - 1) & 1, abort_flag)) {
                    ok = false;
                    break;
                }
                tc_fence_after_sync();
                const uint32_t d = tmem + static_cast<uint32_t>(b * 2 * kMnGroup);
                for (int kb = 0; kb < n_kb; ++kb, ++it) {
                    const int s = it % kMnStages, u = it / kMnStages;
                    if (!mbar_wait(&full[s], u & 1, abort_flag)) {
                        ok = false;
                        break;
                    }
                    tc_fence_after_sync();
                    unsigned char *st = ring + s * kMnStageBytes;
                    const uint64_t ad = umma_desc_k_sw128(st), bd = umma_desc_k_sw128(st + kMnStageBytes / 2);
#pragma unroll
                    for (int k4 = 0; k4 < 4; ++k4)
                        umma_bf16_pair(d, ad + 2 * k4, bd + 2 * k4, idesc, (kb | k4) != 0 ? 1u : 0u);
                    umma_commit_pair(&empty[s]);
                }
                if (ok) umma_commit_pair(&tfull[b]);
            }
            if (!ok) {
                atomicOr(p.err, kErrWaitTimeout);
                mc->abort = 1;
            }
            // every MMA this thread issued has finished before TMEM is freed
            umma_commit_pair_local(final_bar);
            const int never = 0;
            mbar_wait(final_bar, 0, const_cast<volatile int *>(&never));
        }
        __syncwarp();
    } else {
        // ---------------- epilogue ----------------
        griddep_wait();  // the bounds; and the outputs follow the previous kernel
        const int qw = warp & 3, half = (warp - 2) >> 2;
        const unsigned row_in_tile = rank * 128u + 32u * qw + lane;
        int ti = 0;
        for (int item = pair; item < n_items; item += n_pairs, ++ti) {
            const int tile = item / p.groups, g = item - tile * p.groups;
            const int b = ti & 1, ub = ti >> 1;
            if (!mbar_wait(&tfull[b], ub & 1, abort_flag)) {
                if (lane == 0) {
                    atomicOr(p.err, kErrWaitTimeout);
                    mc->abort = 1;
                }
                break;
            }
            tc_fence_after_sync();
            const int64_t row = static_cast<int64_t>(tile) * kMnRows + row_in_tile;
            const bool real = row < p.rows;
            const uint32_t tb = tmem + (static_cast<uint32_t>(32 * qw) << 16) + b * 2 * kMnGroup + half * kMnGroup;
            const int q0 = g * kMnGroup + half * (kMnGroup / 2);
#pragma unroll 1
            for (int c = 0; c < 4; ++c) {  // 32 columns, 16 queries
                uint32_t r[2][16];
                tmem_ld_32x32b_x16(tb + 32 * c, r[0]);
                tmem_ld_32x32b_x16(tb + 32 * c + 16, r[1]);
                tmem_wait_ld();
                float z[16];
#pragma unroll
                for (int i = 0; i < 16; ++i)
                    z[i] = __uint_as_float(r[i / 8][2 * (i % 8)]) + __uint_as_float(r[i / 8][2 * (i % 8) + 1]);
                const int q = q0 + 16 * c;
                if (p.sample != nullptr) {
                    if (real) {
#pragma unroll
                        for (int i = 0; i < 16; ++i) p.sample[(q + i) * p.sample_pitch + row] = z[i];
                    }
                    continue;
                }
                uint32_t in = 0;
                const float4 *t4 = reinterpret_cast<const float4 *>(p.tau_v + q);
#pragma unroll
                for (int i = 0; i < 4; ++i) {
                    const float4 t = t4[i];
                    in |= (z[4 * i] >= t.x ? 1u : 0u) << (4 * i);
                    in |= (z[4 * i + 1] >= t.y ? 1u : 0u) << (4 * i + 1);
                    in |= (z[4 * i + 2] >= t.z ? 1u : 0u) << (4 * i + 2);
                    in |= (z[4 * i + 3] >= t.w ? 1u : 0u) << (4 * i + 3);
                }
                if (!real) in = 0;
                if (__any_sync(0xFFFFFFFFu, in != 0)) {
#pragma unroll
                    for (int i = 0; i < 16; ++i) {
                        if (in >> i & 1u) {
                            const uint64_t key = make_key(z[i], static_cast<uint32_t>(row));
                            if (key >= p.tau[q + i]) {
                                const uint32_t pos = atomicAdd(p.count + q + i, 1u);
                                if (pos < kMnCap) p.cand[static_cast<size_t>(q + i) * kMnCap + pos] = key;
                            }
                        }
                    }
                }
                __syncwarp();
            }
            tc_fence_before_sync();
            __syncwarp();
            if (lane == 0) mbar_arrive_cluster(cluster_map(&tempty[b], 0));
        }
    }

    __syncthreads();
    cluster_sync();  // neither CTA signals the other any more, and its operands are no longer read
    if (warp == 1) {
        tc_fence_after_sync();
        tmem_dealloc_pair(tmem, 512);
    }
}

namespace {

// Keys of the sampled rows of one query: logit z[i] of vocabulary row i * stride.
struct SampleKeys {
    const float *z;
    uint32_t stride;
    __device__ __forceinline__ uint64_t operator[](int i) const {
        return make_key(z[i], static_cast<uint32_t>(i) * stride);
    }
};

}  // namespace

// One CTA per query slot of the block: tau[q] = a key with at least k sampled
// keys at or above it, tau_v[q] its logit (+inf for slots without a query, so
// that none of their logits pass), count[q] = ticket[q] = 0.  The sampled logits are read
// once, into registers; a histogram over the upper half of their range gives
// the bin of the k-th largest, and the smallest logit of that bin and those
// above it is the bound.  Where that would be a bound of more than max_rank
// sampled keys (ties, outliers; many_max_rank), or the sample has more rows than
// the registers hold, a radix select finds the exact k-th key (13.3 us per 512
// queries of 2374 sampled rows).
constexpr int kTauThreads = 512;
template <int PER>
__global__ void __launch_bounds__(kTauThreads, PER <= 8 ? 3 : 1) many_tau_kernel(const float *__restrict__ sample, int64_t pitch, int rows,
                                                               uint32_t stride, int nq, int k, int max_rank, uint64_t *tau,
                                                               float *tau_v, uint32_t *count, uint32_t *ticket) {
    constexpr int kBins = 1024;
    __shared__ uint32_t hist[kBins];
    __shared__ uint32_t range[4];  // lowest, highest ordered logit, the k-th largest's bin (+ 1; 0: crowded), bound
    __shared__ MiscSmem ms;
    griddep_launch_dependents();
    const int q = blockIdx.x, tid = threadIdx.x, lane = tid & 31;
    if (tid == 0) {
        range[0] = 0xFFFFFFFFu;
        range[1] = 0u;
        range[2] = 0u;
        range[3] = 0xFFFFFFFFu;
    }
    for (int i = tid; i < kBins; i += kTauThreads) hist[i] = 0;
    griddep_wait();
    uint64_t t = ~0ull;
    if (q < nq) {  // (the whole CTA)
        const float *z = sample + q * pitch;
        t = 0;
        if (rows <= PER * kTauThreads) {
            uint32_t v[PER], lo = 0xFFFFFFFFu, hi = 0u;
#pragma unroll
            for (int j = 0; j < PER; ++j) v[j] = tid + j * kTauThreads < rows ? order_f32(z[tid + j * kTauThreads]) : 0u;
#pragma unroll
            for (int j = 0; j < PER; ++j) {
                hi = max(hi, v[j]);
                if (tid + j * kTauThreads < rows) lo = min(lo, v[j]);
            }
            lo = __reduce_min_sync(0xFFFFFFFFu, lo);
            hi = __reduce_max_sync(0xFFFFFFFFu, hi);
            __syncthreads();
            if (lane == 0) {
                atomicMin(&range[0], lo);
                atomicMax(&range[1], hi);
            }
            __syncthreads();
            // equal bins of the upper half of the logits' range
            const float top = unorder_f32(range[1]), mid = 0.5f * unorder_f32(range[0]) + 0.5f * top;
            const float scale = top > mid ? kBins / (top - mid) : 0.0f;
            int bin[PER];
#pragma unroll
            for (int j = 0; j < PER; ++j) {
                const float x = unorder_f32(v[j]);
                bin[j] = tid + j * kTauThreads < rows && x >= mid ? min(kBins - 1, static_cast<int>((x - mid) * scale)) : -1;
                if (bin[j] >= 0) atomicAdd(&hist[bin[j]], 1u);
            }
            __syncthreads();
            if (tid < 32) {  // lane l: bins kBins - 1 - 32 l downwards (read rotated: distinct banks)
                const int b0 = kBins - 32 - 32 * lane;
                uint32_t local = 0;
                for (int j = 0; j < 32; ++j) local += hist[b0 + ((j + lane) & 31)];
                uint32_t incl = local;
#pragma unroll
                for (int o = 1; o < 32; o <<= 1) {
                    const uint32_t x = __shfl_up_sync(0xFFFFFFFFu, incl, o);
                    if (lane >= o) incl += x;
                }
                uint32_t run = incl - local;
                const uint32_t uk = static_cast<uint32_t>(k);
                if (run < uk && uk <= incl) {
                    int b = b0 + 31;
                    while (run + hist[b] < uk) run += hist[b--];
                    if (run + hist[b] <= static_cast<uint32_t>(max_rank)) range[2] = static_cast<uint32_t>(b) + 1u;
                }
            }
            __syncthreads();
            if (range[2] != 0) {  // the smallest logit of that bin and those above
                const int b = static_cast<int>(range[2]) - 1;
                lo = 0xFFFFFFFFu;
#pragma unroll
                for (int j = 0; j < PER; ++j)
                    if (bin[j] >= b) lo = min(lo, v[j]);
                lo = __reduce_min_sync(0xFFFFFFFFu, lo);
                if (lane == 0) atomicMin(&range[3], lo);
                __syncthreads();
                t = static_cast<uint64_t>(range[3]) << 32;
            }
        }
        __syncthreads();
        if (t == 0) t = block_radix_threshold(SampleKeys{z, stride}, rows, k, 1, hist, &ms);
    }
    if (tid == 0) {
        const uint32_t hi = static_cast<uint32_t>(t >> 32);
        tau[q] = t;
        // (below order_f32(-FLT_MAX) there are only -inf and NaN patterns)
        tau_v[q] = q >= nq ? __uint_as_float(0x7F800000u) : (hi < 0x00800000u ? __uint_as_float(0xFF800000u) : unorder_f32(hi));
        count[q] = 0;
        ticket[q] = 0;
    }
}

// The best k of the logits of rows [r0, r1) of W against hq, and often a few
// more, to mb.cands; returns how many there are.  fp32 dot products, four rows per warp at a
// time, 16 bytes per lane and row: 20 KB in flight per CTA, four CTAs per SM.
static __device__ __forceinline__ int rescan_rows(const uint16_t *W, int64_t r0, int64_t r1, int d, int d_pad,
                                               const float *hq, int k, const MergeBufs &mb, MiscSmem *ms) {
    constexpr int kWarps = kThreads / 32, kRows = 4;
    constexpr int kRound = kMergeCandCap / 2;  // rows between cut-backs; k <= kMnMaxK keys stay
    static_assert(kMnMaxK <= kRound, "a round's keys and those kept fit the buffer");
    const int tid = threadIdx.x, lane = tid & 31, warp = tid >> 5;
    const int C = d_pad >> 3;
    const bool vec = (reinterpret_cast<uintptr_t>(hq) & 15u) == 0;
    uint64_t bound = 1;
    if (tid == 0) ms->n_cand = 0;
    __syncthreads();
    int n = 0;
    for (int64_t a = r0; a < r1; a += kRound) {
        const int rows = static_cast<int>(min(static_cast<int64_t>(kRound), r1 - a));
        const uint4 *Wa = reinterpret_cast<const uint4 *>(W) + a * C;
        for (int b = kRows * warp; b < rows; b += kRows * kWarps) {
            float acc[kRows] = {};
#pragma unroll 1
            for (int c = lane; c < C; c += 32) {
                uint4 w[kRows];
#pragma unroll
                for (int i = 0; i < kRows; ++i)
                    w[i] = __ldg(Wa + static_cast<int64_t>(min(b + i, rows - 1)) * C + c);
                float x[8];
                if (vec && 8 * c + 8 <= d) {
                    const float4 lo = __ldg(reinterpret_cast<const float4 *>(hq) + 2 * c);
                    const float4 hi = __ldg(reinterpret_cast<const float4 *>(hq) + 2 * c + 1);
                    x[0] = lo.x, x[1] = lo.y, x[2] = lo.z, x[3] = lo.w;
                    x[4] = hi.x, x[5] = hi.y, x[6] = hi.z, x[7] = hi.w;
                } else {
#pragma unroll
                    for (int e = 0; e < 8; ++e) x[e] = 8 * c + e < d ? __ldg(hq + 8 * c + e) : 0.0f;
                }
#pragma unroll
                for (int i = 0; i < kRows; ++i) {
                    acc[i] = fmaf(bf16_lo(w[i].x), x[0], acc[i]);
                    acc[i] = fmaf(bf16_hi(w[i].x), x[1], acc[i]);
                    acc[i] = fmaf(bf16_lo(w[i].y), x[2], acc[i]);
                    acc[i] = fmaf(bf16_hi(w[i].y), x[3], acc[i]);
                    acc[i] = fmaf(bf16_lo(w[i].z), x[4], acc[i]);
                    acc[i] = fmaf(bf16_hi(w[i].z), x[5], acc[i]);
                    acc[i] = fmaf(bf16_lo(w[i].w), x[6], acc[i]);
                    acc[i] = fmaf(bf16_hi(w[i].w), x[7], acc[i]);
                }
            }
            uint64_t key = 0;
#pragma unroll
            for (int i = 0; i < kRows; ++i) {
                float z = acc[i];
#pragma unroll
                for (int o = 16; o >= 1; o >>= 1) z += __shfl_xor_sync(0xFFFFFFFFu, z, o);
                if (lane == i && b + i < rows) key = make_key(z, static_cast<uint32_t>(a) + static_cast<uint32_t>(b + i));
            }
            if (key >= bound) mb.cands[atomicAdd(&ms->n_cand, 1)] = key;
        }
        __syncthreads();
        n = ms->n_cand;
        __syncthreads();  // read by all before the next round adds to it
        if (n > k && (n > kRound || a + kRound >= r1)) {  // keep the best k
            const uint64_t T = block_radix_threshold(SmemKeys{mb.cands}, n, k, 1, mb.hist, ms);
            if (tid == 0) ms->n_win = 0;
            __syncthreads();
            for (int i = tid; i < n; i += kThreads)
                if (mb.cands[i] >= T) mb.win[atomicAdd(&ms->n_win, 1)] = mb.cands[i];
            __syncthreads();
            for (int i = tid; i < k; i += kThreads) mb.cands[i] = mb.win[i];
            bound = T;
            n = k;
            if (tid == 0) ms->n_cand = k;
            __syncthreads();
        }
    }
    return n;
}

// The buffers of a merge in mem (SmemLayout::merge_fixed_bytes()).
static __device__ __forceinline__ MergeBufs merge_bufs(unsigned char *mem) {
    MergeBufs mb;
    mb.pref = reinterpret_cast<uint64_t *>(mem);
    mb.cands = mb.pref + kMergePrefixCap;
    mb.win = mb.cands + kMergeCandCap;
    mb.counts = reinterpret_cast<int *>(mb.win + 1024);
    mb.offsets = mb.counts + kMaxLists;
    mb.hist = reinterpret_cast<uint32_t *>(mb.offsets + kMaxLists);
    return mb;
}

// Whether a query's list of n candidates holds its top k (too many were not
// kept; too few are logits that are not numbers).
static __device__ __forceinline__ bool complete(uint32_t n, int k) {
    return n >= static_cast<uint32_t>(k) && n <= kMnCap;
}

// Query q's row of the sparse tensor, -inf so far; nullptr without one.
static __device__ __forceinline__ float *fill_sparse(const MnFinalParams &p, int q) {
    if (p.sparse == nullptr) return nullptr;
    float *sp = p.sparse + q * p.V;
    for (int64_t i = threadIdx.x; i < p.V; i += kThreads) sp[i] = __uint_as_float(0xFF800000u);
    return sp;
}

// The queries without a complete list, recomputed from all rows.  All CTAs of
// the launch share the work: kMnCap / k slices of the rows per such query, the
// k best of each slice to the query's own list, and the CTA that finishes the
// last slice ranks them (a ticket; nobody waits).
static __device__ __noinline__ void rescan_queries(const MnFinalParams &p, unsigned char *mem, MiscSmem *ms) {
    __shared__ uint16_t missed[kMnBlock];
    __shared__ int n_missed, last;
    const MergeBufs mb = merge_bufs(mem);
    const int tid = threadIdx.x, lane = tid & 31, k = p.k;
    if (tid < 32) {  // in the same order in every CTA
        int n = 0;
        for (int i0 = 0; i0 < p.nq; i0 += 32) {
            const bool m = i0 + lane < p.nq && !complete(p.count[i0 + lane], k);
            const unsigned mask = __ballot_sync(0xFFFFFFFFu, m);
            if (m) missed[n + __popc(mask & ((1u << lane) - 1u))] = static_cast<uint16_t>(i0 + lane);
            n += __popc(mask);
        }
        if (lane == 0) n_missed = n;
    }
    __syncthreads();
    const int slices = min(kMnCap / k, 256), tasks = slices * n_missed;
    const int64_t share = (p.V + slices - 1) / slices;
    for (int t = blockIdx.x; t < tasks; t += gridDim.x) {
        const int s = t / n_missed, q = missed[t - s * n_missed];
        const int64_t r0 = min(p.V, s * share), r1 = min(p.V, r0 + share);
        const int n = rescan_rows(p.W, r0, r1, p.d, p.d_pad, p.h + static_cast<int64_t>(q) * p.d, k, mb, ms);
        uint64_t *list = p.cand + static_cast<size_t>(q) * kMnCap;
        for (int i = tid; i < k; i += kThreads) list[s * k + i] = i < n ? mb.cands[i] : 0ull;
        __syncthreads();  // orders the slice's keys before thread 0's ticket
        if (tid == 0) {
            last = atomic_add_acq_rel_gpu(p.ticket + q, 1u) == static_cast<uint32_t>(slices - 1) ? 1 : 0;
            ms->n_cand = 0;
        }
        __syncthreads();
        if (last) {
            float *sp = fill_sparse(p, q);
            for (int i = tid; i < slices * k; i += kThreads) {
                const uint64_t x = __ldcg(reinterpret_cast<const unsigned long long *>(list) + i);
                if (x != 0) mb.cands[atomicAdd(&ms->n_cand, 1)] = x;
            }
            __syncthreads();
            block_topk_to_output(mb.cands, ms->n_cand, k, mb, ms, p.out_idx + static_cast<int64_t>(q) * k,
                                 p.out_logits + static_cast<int64_t>(q) * k, sp);
        }
        __syncthreads();  // the buffers are free for the next task
    }
}

// One CTA per query: the exact top-k of its candidates, best first, and its
// row of the sparse tensor; then the queries whose lists overflowed, together.
// One such query of 512 adds 0.23 ms at 151936 x 1024, k = 2 (33 ms when its own
// CTA recomputed it alone, two bytes at a time) and 2.7 ms at 128256 x 3072, k =
// 50, 40 slices (80 ms); all 512 of them take 28 and 124 ms (43 and 234 ms).
// (Four CTAs per SM: with the registers that the recomputation would like, two
// would fit, and every block pays for that.)
__global__ void __launch_bounds__(kThreads, 4) many_final_kernel(const __grid_constant__ MnFinalParams p) {
    extern __shared__ __align__(16) unsigned char fin_smem[];
    __shared__ MiscSmem ms;
    griddep_launch_dependents();
    griddep_wait();
    const int q = blockIdx.x, tid = threadIdx.x, k = p.k;
    const uint32_t n = p.count[q];
    bool miss = false;
    for (int i = tid; i < p.nq; i += kThreads) miss |= !complete(p.count[i], k);
    static_assert(kMnCap <= kMergeCandCap, "a query's candidates are ranked in shared memory");
    if (complete(n, k)) {
        float *sp = fill_sparse(p, q);
        const MergeBufs mb = merge_bufs(fin_smem);
        const uint64_t *list = p.cand + static_cast<size_t>(q) * kMnCap;
        for (int i = tid; i < static_cast<int>(n); i += kThreads)
            mb.cands[i] = __ldcg(reinterpret_cast<const unsigned long long *>(list) + i);
        __syncthreads();
        block_topk_to_output(mb.cands, static_cast<int>(n), k, mb, &ms, p.out_idx + static_cast<int64_t>(q) * k,
                             p.out_logits + static_cast<int64_t>(q) * k, sp);
    }
    if (__syncthreads_or(miss ? 1 : 0)) rescan_queries(p, fin_smem, &ms);
}

cudaError_t launch_tc_many(const CUtensorMap &mapW, const CUtensorMap &mapH, const MnParams &p, int sms,
                           cudaStream_t stream) {
    static bool configured[64] = {};
    int dev = 0;
    cudaError_t e = cudaGetDevice(&dev);
    if (e != cudaSuccess) return e;
    if (dev < 0 || dev >= 64) return cudaErrorInvalidDevice;
    if (!configured[dev]) {
        e = cudaFuncSetAttribute(tc_many_kernel, cudaFuncAttributeMaxDynamicSharedMemorySize, kMnSmem);
        if (e == cudaSuccess)
            e = cudaFuncSetAttribute(many_final_kernel, cudaFuncAttributeMaxDynamicSharedMemorySize,
                                     SmemLayout::merge_fixed_bytes());
        if (e != cudaSuccess) return e;
        configured[dev] = true;
    }
    int64_t pairs = (p.rows + kMnRows - 1) / kMnRows * p.groups;
    if (pairs > sms / 2) pairs = sms / 2;
    return launch_pdl(tc_many_kernel, dim3(static_cast<unsigned>(2 * pairs)), dim3(kMnThreads), kMnSmem, stream, mapW,
                      mapH, p);
}

cudaError_t launch_many_tau(const float *sample, int64_t pitch, int rows, int stride, int nq, int slots, int k,
                            uint64_t *tau, float *tau_v, uint32_t *count, uint32_t *ticket, cudaStream_t stream) {
    const auto kern = rows <= 8 * kTauThreads ? many_tau_kernel<8> : many_tau_kernel<32>;
    return launch_pdl(kern, dim3(static_cast<unsigned>(slots)), dim3(kTauThreads), 0, stream, sample, pitch, rows,
                      static_cast<uint32_t>(stride), nq, k, many_max_rank(k), tau, tau_v, count, ticket);
}

cudaError_t launch_many_final(const MnFinalParams &p, cudaStream_t stream) {
    return launch_pdl(many_final_kernel, dim3(static_cast<unsigned>(p.nq)), dim3(kThreads),
                      SmemLayout::merge_fixed_bytes(), stream, p);
}

}  // namespace vie
