// vie_tc_many.cuh - the output head for many queries at once (a Recall@k
// ground truth over thousands of hidden states, prefill-sized batches): the
// exact top-k as a filtered GEMM instead of one pass over W per 64 queries.
//
// Per block of up to kMnBlock queries, five launches:
//   prep    the hi/lo bf16 query matrix (as on the batched path);
//   sample  the GEMM below on every s-th row of W, logits written out;
//   tau     per query, a key with at least k sampled keys at or above it (the
//           k-th largest, or one of little higher rank): a bound on the k-th
//           key of the whole vocabulary;
//   main    the GEMM on all rows; a logit whose key is at least the query's
//           tau is appended to its candidate list (about k s of them, s chosen
//           so that kMnCap holds them), everything else stays on the chip;
//   final   per query, the exact top-k of its candidates.
// The sample takes every s-th row of the total order's index range, and tau is
// a key (logit, then row), so neither ties nor clusters of neighbouring rows
// make many candidates; a query whose list overflows all the same (kMnCap)
// is recomputed from all rows by the CTAs of the final launch.  20000 queries,
// 151936 x 1024, k = 2: 22.0 ms in passes of 64 queries, 9.0 ms here (per 512
// queries: main 194 us, 1.64 PFLOP/s; the other four launches ~30 us).
//
// The GEMM runs on CTA pairs (tcgen05 cta_group::2): M = 256 rows of W, half
// per CTA, times N = 256 columns, 128 queries as hi and lo. Each CTA stages its
// half of both operands (32 KB per 64 columns of K), so a stage feeds twice
// the arithmetic of a single CTA's tile at the same bytes; the accumulators
// (2 x 256 TMEM columns) are double buffered. A logit is the sum of its two
// columns, each accumulated over K in the same steps as on the batched path.
//   warp 0     TMA producer (both CTAs; bytes counted on the leader's barrier);
//   warp 1     TMEM allocator; the leader's lane 0 issues every MMA, commits
//              free the stage in both CTAs;
//   warps 2-9  epilogue: TMEM lane quarter w % 4, half of the columns each.
// All waits are bounded.
#pragma once

#include <cuda.h>
#include <cstdint>

#include "vie_plan.h"

namespace vie {

constexpr int kMnGroup = 128;      // queries of a tile (hi and lo: 256 columns)
constexpr int kMnBlock = 512;      // queries of a block of launches, at most
constexpr int kMnRows = 256;       // rows of a tile (a CTA pair)
constexpr int kMnStages = 6;
constexpr int kMnStageBytes = 2 * 128 * 128;  // per CTA: 128 rows of W and of the query matrix
constexpr int kMnEpiWarps = 8;
constexpr int kMnThreads = 32 * (2 + kMnEpiWarps);
constexpr uint32_t kMnSmem = 1024 + kMnStages * kMnStageBytes + 1024;  // barriers, ring, its alignment

struct MnParams {
    int64_t rows;          // rows of the W operand: V, or those of the sample
    int32_t d_pad;
    int32_t groups;        // query groups of the block
    float *sample;         // the sample launch: logits [query][sample_pitch]; else nullptr
    int64_t sample_pitch;
    const uint64_t *tau;   // main: [query] bound keys and their logits
    const float *tau_v;
    uint64_t *cand;        // [query][kMnCap] keys
    uint32_t *count;       // [query]
    uint32_t *err;
};

struct MnFinalParams {
    uint64_t *cand;         // [query][kMnCap] keys
    const uint32_t *count;  // [query] candidates that reached the bound
    uint32_t *ticket;       // [query] slices finished, 0 before the launch
    int32_t nq, k;
    const uint16_t *W;      // [V][d_pad] bf16 bits
    int64_t V;
    int32_t d, d_pad;
    const float *h;         // [nq][d]
    int32_t *out_idx;       // [nq][k]
    float *out_logits;      // [nq][k]
    float *sparse;          // [nq][V] or nullptr
};

}  // namespace vie
