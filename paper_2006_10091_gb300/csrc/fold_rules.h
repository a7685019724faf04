// fold_rules.h -- which primes and which sums take the folded and split
// arithmetic of he_common.cuh and ks_fused.cuh.  Plain C++ (host and device), so
// that the CPU tests compile these rules themselves and check each bound.
#pragma once
#include <stdint.h>

#ifdef __CUDACC__
#define HE_RULE __host__ __device__ __forceinline__
#else
#define HE_RULE inline
#endif

inline uint32_t bit_length(uint64_t x) { return x ? 64 - __builtin_clzll(x) : 0; }

// delta = 2^k - q of a prime q of k bits whose folds apply, else 0: 33 <= k <= 60
// and delta below 2^28 and 2^((2k-4)/3) (both are below 2^(k-13) there).
inline uint32_t fold_delta(uint64_t q) {
  const uint32_t k = bit_length(q);
  if (k < 33 || k > 60) return 0;
  const uint64_t d = (1ull << k) - q;
  const uint32_t lim = (2 * k - 4) / 3 < 28 ? (2 * k - 4) / 3 : 28;
  return d >> lim ? 0 : (uint32_t)d;
}

// Butterflies as split products (mul_split): values must stay below 2^46.
constexpr uint32_t kSplitMaxBits = 40;

// Products a split sum may hold.  split3_residue's last fold leaves less than
// 2q up to 3470 of them (35 bits, delta at its bound: the narrowest prime for
// its delta).  The callers' own limits keep below this (static assertions there):
// a comparison in the kernels moved ks_row_rot's registers, a stage of seven
// rotations at N = 2^14 1220 -> 1229 us.
constexpr uint32_t kSplit3Terms = 1024;

// Whether nterms products of residues below 2^k (and part 0's term, below
// 1.01 times as much) can be summed as split sums; nterms <= kSplit3Terms.
HE_RULE bool split3_fits(uint32_t k, uint32_t nterms) {
  uint32_t bits = 0;
  for (uint32_t x = nterms + 2; x; x >>= 1) ++bits;
  return 2 * ((k + 1) / 2) + 2 + bits <= 64;
}

// Whether the conversion of cnt sources below 2^src_bits to q runs as
// conv_split_tile: the sum (plus 3q for ModDown's lift) stays below 2^64 and its
// fold below 2^(k+5) (2^(k+3) for the split products' primes, 2q for the corrected
// transforms'), so that the transform's values stay in range.
inline bool conv_split_ok(uint64_t q, uint32_t cnt, uint32_t src_bits) {
  typedef unsigned __int128 u128;
  const uint32_t k = bit_length(q), e = (k + 1) / 2;
  const uint64_t delta = fold_delta(q);
  if (!delta || cnt < 1 || cnt > 5 || src_bits > 60) return false;
  const u128 rho = (u128)delta << (2 * e - k);
  u128 most = (u128)1 << src_bits;
  if (cnt > 1) {
    const u128 a = (u128)(2 * cnt) << (30 + e), b = (u128)(2 * cnt) << (30 + k - e);
    if (b >> 64) return false;
    most = a + ((u128)1 << (2 * e)) + ((b >> e) + 1) * rho;
  }
  most += 3 * (u128)q;
  if (most >> 64) return false;
  const u128 folded = ((u128)1 << k) + (most >> k) * delta;
  return folded <= (k <= kSplitMaxBits ? (u128)1 << (k + 3) : q < (1ull << 58) ? (u128)1 << (k + 5) : 2 * (u128)q);
}

