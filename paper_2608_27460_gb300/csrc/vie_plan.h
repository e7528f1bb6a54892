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
// CTAs: one per tile, or four (of 32 rows each) where one from every CTA would
// be too few for k; none (0) where neither gives k of them.
constexpr int tc_bound_blocks(int slots, int k, int G) {
    const int b = 2 * k <= G || !bound_words_fit(slots, 4) ? 1 : 4;
    return b * G >= k && b * G <= kBoundMax && bound_words_fit(slots, b) ? b : 0;
}
static_assert(bound_words_fit(64, 4) && bound_words_fit(8, 8), "the widest tensor-core and streaming launches");

}  // namespace vie
