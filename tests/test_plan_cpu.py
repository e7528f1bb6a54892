"""Launch-planning rules that need no GPU (csrc/vie_plan.h), compiled and
enumerated here over every shape a call can take."""
import os
import shutil
import subprocess

import pytest

ROOT = os.path.dirname(os.path.dirname(os.path.abspath(__file__)))
CSRC = os.path.join(ROOT, "paper_2608_27460_gb300", "csrc")


def run_cpp(tmp_path, body):
    """Compiles `body` as main() behind vie_plan.h and returns its output lines."""
    gxx = shutil.which("g++")
    if gxx is None:
        pytest.skip("no g++")
    src, exe = tmp_path / "plan.cpp", tmp_path / "plan"
    src.write_text('#include <cstdio>\n#include <initializer_list>\n#include "vie_plan.h"\nusing namespace vie;\nint main() {\n' + body + "\n}\n")
    subprocess.run([gxx, "-std=c++17", "-O1", "-Wall", "-Werror", "-I", CSRC, str(src), "-o", str(exe)], check=True)
    return subprocess.run([str(exe)], check=True, capture_output=True, text=True).stdout.split("\n")[:-1]


def test_shared_bound_words_stay_within_their_room(tmp_path):
    """A tensor-core launch of `slots` query slots publishes slots * blocks
    words per CTA; what lies behind the kBoundWords of a handle is the query
    matrix the same launch reads.  Every tile, k and number of CTAs (one per 64
    rows at most) and vocabularies of up to ten tiles per CTA: 64 slots take k up
    to 64, the others up to 128.  Where a bound is used, the CTAs that have a tile
    publish at least k words; it is used wherever four of each are k, but for the smallest k of
    64 slots and of rows of odd sectors."""
    out = run_cpp(tmp_path, """
    for (int slots : {4, 8, 16, 32, 64})
        for (int k = 1; k <= (slots == 64 ? 64 : 128); ++k)
            for (int G = 1; G <= 1024; ++G)
                for (int V : {64 * G - 63, 64 * G - 5, 64 * G, 64 * G + 37, 128 * G - 127, 128 * G - 1, 1280 * G}) {
                    const int b = tc_bound_blocks(slots, k, G, V, 2048);
                    int words = 0;  // row block r of 32 (b = 4) or 128 rows (b = 1), the first tile of each CTA
                    words = b == 4 ? (V + 31) / 32 : (V + 127) / 128;
                    words = words < b * G ? words : b * G;
                    if (b != 0 && b != 1 && b != 4) std::printf("blocks %d %d %d: %d\\n", slots, k, G, b);
                    if (slots * b > kBoundWords) std::printf("words %d %d %d: %d\\n", slots, k, G, b);
                    if (b * G > kBoundMax) std::printf("count %d %d %d: %d\\n", slots, k, G, b);
                    if (b != 0 && words < k) std::printf("few %d %d %d %d: %d\\n", slots, k, G, V, b);
                    const int most = (V + 31) / 32 < 4 * G ? (V + 31) / 32 : 4 * G;
                    if (b == 0 && (slots < 64 || k > 1) && most >= k && 4 * G <= kBoundMax) std::printf("unused %d %d %d\\n", slots, k, G);
                    if (tc_bound_blocks(slots, k, G, V, 2000) != (slots > 4 && k <= 3 ? 0 : b)) std::printf("pitch %d %d\\n", slots, k);
                }""")
    assert not out, out[:10]


def test_candidates_of_many_queries_seldom_overflow(tmp_path):
    """The bound of a query is its r-th largest sampled logit, r at most the rank
    the bounds kernel accepts.  More than `cap` keys reach it exactly when fewer
    than r of the cap best keys were sampled, each with probability 1 / stride:
    at most one query in 10^6, for every k."""
    binom = pytest.importorskip("scipy.stats").binom
    out = run_cpp(tmp_path, """
    for (int k = 1; k <= kMnMaxK; ++k)
        std::printf("%d %d %d %d\\n", k, 8 << many_stride_log2(k), many_max_rank(k), kMnCap);""")
    assert len(out) == 128
    for line in out:
        k, stride, rank, cap = map(int, line.split())
        assert rank >= k, line
        assert binom.cdf(rank - 1, cap, 1.0 / stride) <= 1e-6, line
