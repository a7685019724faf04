// tile_pairs.h -- the tile-shape pairs of the two-pass transforms and of the
// fused key-switching kernels: per ring size N = 2^12 .. 2^16 three pairs
// (column pass bits, rows per tile | row pass bits, rows per tile).  Plain C++,
// read by the CPU tests too.
#pragma once

namespace he {

struct TilePair {
  int m1, k1, m2, k2;
};

// In the order of the tuning knob "ntt_shape": programs keep its values (a
// tuning that he_autotune found, say), so a pair never moves.
constexpr TilePair kTilePairs[5][3] = {
    {{6, 5, 6, 5}, {5, 6, 7, 4}, {3, 8, 9, 2}},   // N = 2^12
    {{7, 4, 6, 5}, {6, 5, 7, 4}, {4, 7, 9, 2}},   // N = 2^13
    {{7, 4, 7, 4}, {8, 3, 6, 5}, {5, 6, 9, 2}},   // N = 2^14
    {{8, 4, 7, 4}, {7, 4, 8, 3}, {6, 5, 9, 2}},   // N = 2^15
    {{8, 4, 8, 3}, {7, 4, 9, 2}, {6, 5, 10, 1}},  // N = 2^16
};

// A context's pair until it is set or tuned, the one that measured fastest where
// they differ: the gradient step at N = 2^14 63.2 ms (pairs 0 and 1: 66.0 and
// 66.9), a weighted sum at N = 2^15 106 us (107 and 114), eight multiplications
// at N = 2^16 with 24 limbs 2.98 ms (pair 1 3.00; pair 0, a 4096-word column tile
// whose ModUp constants do not fit beside it, 3.94).
constexpr int kDefaultPair[5] = {0, 0, 2, 1, 2};

constexpr int default_pair(int log_n) { return log_n >= 12 && log_n <= 16 ? kDefaultPair[log_n - 12] : 0; }

template <int LOG_N, int SHAPE>
struct PairOf {
  static constexpr int m1 = kTilePairs[LOG_N - 12][SHAPE].m1, k1 = kTilePairs[LOG_N - 12][SHAPE].k1;
  static constexpr int m2 = kTilePairs[LOG_N - 12][SHAPE].m2, k2 = kTilePairs[LOG_N - 12][SHAPE].k2;
};

// f(PairOf<LOG_N, shape>()) for a runtime shape.
template <int LOG_N, class F>
auto with_pair(int shape, F f) {
  return shape == 1 ? f(PairOf<LOG_N, 1>()) : shape == 2 ? f(PairOf<LOG_N, 2>()) : f(PairOf<LOG_N, 0>());
}

}  // namespace he
