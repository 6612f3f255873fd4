// How the rotary append divides its tokens among CTAs (kv_append_rope.cu); host arithmetic only.
#pragma once
#include <algorithm>
#include <cstddef>

namespace asynclm {

constexpr int kRopeThreads = 256, kRopeTokens = 20;      // of a CTA, at most
constexpr int kRopeWave = 148 * 3;                // CTAs of that many threads that run at once
constexpr int kRopeFirstCtas = 148 * 4;           // a wave and a little: see angles_first in the kernel

// A (token, head) row takes head_dim / 16 threads; `heads` are the K heads and, where queries are rotated, the Q heads.
inline int rope_threads(int tokens, int heads, int head_dim) {
    return std::min((tokens * heads * (head_dim / 16) + 31) / 32 * 32, kRopeThreads);
}

// 64 angles and a slot for each token.  (With room for 20 in every CTA, an SM held 10 of the small ones that many tokens of few heads
// make: 65 536 tokens of 4 heads of 64, keys only, 41.5 us -> 51.6.)
inline size_t rope_smem(int tokens) { return (size_t)tokens * (64 * 16 + 8); }

// Tokens of a CTA.  One wave takes about as long as its CTAs, so as many as fill a wave, up to 20.  (us a launch from a graph, with one
// token for each 296 and at most four | so, 32/8 heads, queries rotated: 450 tokens 5.2 | 4.7, 1200 8.9 | 7.8, 2048 15.2 | 12.0, 4096
// 24.2 | 21.8, 8192 42.4 | 39.6, 8880 45.5 | 42.3; at head_dim 64 6000 20.6 | 17.0; 6000 of 8/1 heads 8.9 | 6.8.)
// One instead of two and four instead of five where that makes small CTAs of which an SM holds four, with nearly all lanes at work (two | one:
// 520 tokens of 32/8 heads of 64 3.4 | 2.95, of 16/2 heads 3.4 | 2.95, 4/4 heads of 64 keys only 2.1 | 1.9; five | four: 2000 of 4/4 heads of
// 64 3.2 | 2.9; two instead of three and three instead of four: 0.95 to 1.08 of the time).
// Beyond 20 tokens a CTA there are several waves, whose CTAs do not start together, and longer ones are no gain by themselves: four,
// or eight where wide rows or many tokens make it (four | eight | what fills two, three or more waves evenly: 9000 tokens of 32/8 heads
// 46.9 | 47.2 | 46.6, 9500 49.2 | 50.3 | 48.6, 16384 80.6 | 79.8 | 80.3, 65536 306 | 299 | 302, 11 000 56.1 | - | 56.4; 32/8 heads of 64 9500
// 30.4 | 27.9 | 27.7, 65536 185 | 163 | 164; 8/2 heads of 64 9500 12.1 | 12.6 | 12.0, 65536 78 | 81 | 70; 4/4 heads of 64 9500 11.2 | 11.9 |
// 12.1, 16384 17.4 | 19.8 | 18.6).
inline int rope_tokens(int total_q, int heads, int head_dim) {
    const int row_threads = heads * (head_dim / 16);
    const int tokens = std::max(1, (total_q + kRopeWave - 1) / kRopeWave);
    if (tokens > kRopeTokens) return row_threads < 64 || (row_threads > 160 && total_q < 14000) ? 4 : 8;
    if (tokens == 2 || tokens == 5) {
        const int fewer = tokens - 1, threads = rope_threads(fewer, heads, head_dim), idle = threads - fewer * row_threads;
        if ((total_q + fewer - 1) / fewer <= kRopeFirstCtas && threads <= 160 && (threads == 32 || 8 * idle <= threads)) return fewer;
    }
    return tokens;
}

}  // namespace asynclm
