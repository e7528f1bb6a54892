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
// CTAs and so many tiles of W: one of each CTA's first tile, or four (of 32
// rows each) where one from every CTA with a tile would be fewer than 2 k; none
// (0) where four give less than k and a quarter: the bound then lies so low, or
// is never reached, that waiting for it costs more than it saves (V = 2000, 16
// tiles, 64 maxima, b = 4: k = 50 39.8 us without and 17.3 with, k = 64 45.3
// and 48.5, k = 65, where there are too few, 44.7 and 56.2).
constexpr int tc_bound_blocks(int slots, int k, int G, int64_t tiles) {
    const int n = tiles < G ? static_cast<int>(tiles) : G;  // CTAs that publish
    const int b = 2 * k <= n || !bound_words_fit(slots, 4) ? 1 : 4;
    return 4 * b * n >= 5 * k && b * G <= kBoundMax && bound_words_fit(slots, b) ? b : 0;
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
