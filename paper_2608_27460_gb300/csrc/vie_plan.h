// vie_plan.h - rules by which a call's launches are planned that need nothing
// of CUDA: plain constexpr C++, shared by the host code and the kernels.
#pragma once

#include <cstdint>

namespace vie {

// ---- the shared bound's words ----
// Each CTA of a launch publishes, per query slot, `blocks` maxima for the bound
// that all CTAs share: word [slot][cta][block] of the handle's scratch, so a
// launch of `slots` query slots uses slots * blocks words per CTA.  The query
// matrix lies behind those words, so no launch may use more than there are.
constexpr int kBoundMax = 1280;   // maxima behind one query's bound, at most
constexpr int kBoundWords = 256;  // words per CTA: 64 slots x 4 on the tensor-core path, 8 x 8 streaming

constexpr bool bound_words_fit(int slots, int blocks) { return slots * blocks <= kBoundWords; }

// Maxima per CTA and query of a tensor-core launch of `slots` query slots on G
// CTAs, V rows of W in tiles of 128: one of each CTA's first tile, or four (of
// 32 rows each) where G is below 2 k (evaluating four times the words is slower
// where one will do: 12000 rows, 64 queries, k = 50: 32.5 us with one, 54.5 with
// four); none (0) where the rows do not give k of them, which every launch
// would wait for in vain.
// None either where k is so small that a list fills in a handful of insertions
// and starting all CTAs in step costs more: 64 slots at k = 1 (without / with the
// bound: 262144 x 1152 106.5 / 109.7 us, 151936 x 1024 65.5 / 67.6), and up to
// k = 3 where a row's `pitch` bytes are no multiple of a 32-byte sector, so that
// each box of the query matrix, which CTAs in step read at once, takes more of
// them (100003 x 1000, 64 queries: k = 1 57.8 / 68.4, k = 3 60.2 / 69.1, k = 8 68.7 /
// 68.6; e4m3, 32 queries: 41.3 / 48.5, 43.9 / 48.6, 52 without at k = 8 / 48.7; the
// 4-slot tile never waits for the bound and keeps it).
constexpr int tc_bound_blocks(int slots, int k, int G, int64_t V, int64_t pitch) {
    if ((slots == 64 && k == 1) || (slots > 4 && k <= 3 && pitch % 32 != 0)) return 0;
    const int b = 2 * k <= G || !bound_words_fit(slots, 4) ? 1 : 4;
    const int64_t blocks = b == 1 ? (V + 127) / 128 : (V + 31) / 32;  // words there can be
    const int64_t words = blocks < b * G ? blocks : b * G;
    return words >= k && b * G <= kBoundMax && bound_words_fit(slots, b) ? b : 0;
}
static_assert(bound_words_fit(64, 4) && bound_words_fit(8, 8), "the widest tensor-core and streaming launches");

// ---- many queries: the sample ----
constexpr int kMnCap = 2048;   // candidates kept per query
constexpr int kMnMaxK = 128;

// The sample takes every (8 << i)-th row, 64 at most.  A query's bound is its
// r-th largest sampled logit, r >= k, and its candidates are the keys at or above
// that: r times the stride on average, and more than kMnCap where fewer than r of
// the kMnCap best keys were sampled, a binomial tail.  The largest r per stride
// for which that happens to at most one query in 10^6:
constexpr int kMnMaxRank[4] = {188, 79, 30, 9};
constexpr int many_stride_log2(int k) { return k <= 8 ? 3 : (k <= 20 ? 2 : (k <= 64 ? 1 : 0)); }
// The largest rank the bounds kernel accepts: its histogram finds the bin of the
// k-th largest, and the smallest logit of that bin serves when few keys share it.
constexpr int many_max_rank(int k) {
    const int slack = k + k / 4 + 4, most = kMnMaxRank[many_stride_log2(k)];
    return slack < most ? slack : most;
}

}  // namespace vie
