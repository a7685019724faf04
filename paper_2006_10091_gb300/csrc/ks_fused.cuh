// ks_fused.cuh -- hybrid key switching with ModUp fused into the NTT's first
// pass and the key inner product fused into its second pass (N = 2^12 ..
// 2^16).  Same arithmetic and the same residues as the unfused sequence in
// ops.cu (iNTT, k_modup, NTT, k_inner_product); what it saves is the round
// trips of the converted digits through memory:
//  * ks_modup_col: a CTA of digit j and target limb t builds its column tile
//    straight from the coefficient-form input (the digit's limbs, converted
//    to prime t as in k_modup) and runs the column pass; the ModUp output is
//    never written;
//  * ks_row_rot: a CTA of target limb t and two rows finishes the row pass of
//    every digit's tile (or, on the digit's own limb, reads the input as it
//    is), keeps the tiles in shared memory and adds their products with the
//    key polynomials of each rotation (a plain key switch is one rotation by
//    the identity); the transformed digits are never written.  The products
//    are summed as split sums of 32 x 32 -> 64-bit products on primes that
//    allow it (mac_split3) and as 128-bit multiply-accumulates otherwise.
#pragma once
#include <algorithm>
#include <atomic>
#include "he_ops.h"
#include "ntt2.cuh"

namespace he {

// Dynamic shared memory the conversion kernels may take.
constexpr size_t kConvSmemMax = 200 * 1024;
// Largest grid of the row pass that gives each ciphertext four digit groups.
// (One multiplication at N = 2^12 54 -> 47 us, sixteen 66 -> 61, whose grid is 256.)
constexpr size_t kDigitGroupCtas = 304;
// Shared memory of the hoisted rotate-and-sum's row pass (every digit's tile).
constexpr size_t kRotSmemMax = 200 * 1024;

struct KsFusedArgs {
  const uint64_t* d;     // input, evaluation form: count x [level][N] at d_stride
  const uint64_t* d2c;   // input, coefficient form: count x [level][N]
  uint64_t* ext;         // column-pass outputs: count x [beta][nt][N]
  uint64_t* acc;         // accumulators: count x [2][nt][N]
  const uint64_t* evk;   // [beta_top][2][np][N]
  uint64_t d_stride;
  uint64_t gal;            // d is read through the automorphism X -> X^gal (0: none)
  uint32_t level, alpha, beta, L, np, nt;
  const PrimeDev* primes;
  const ulonglong2* tw;
  const ulonglong2* itw;   // inverse twiddles
  int half;                // d2c holds the inverse transform's row pass only (ks_modup_col_all finishes it)
  uint32_t splits;         // CTAs of ks_modup_col_all that share one digit and tile's target limbs
  const uint64_t* consts;  // ModUp constant tables
  uint32_t lo[HE_MAX_PRIMES], cnt[HE_MAX_PRIMES];
  uint64_t off[HE_MAX_PRIMES];
};

__host__ __device__ __forceinline__ uint32_t ks_prime(uint32_t t, uint32_t level, uint32_t L) {
  return t < level ? t : L + t - level;
}

// The basis conversion of one tile into shared memory, y = sum over u < CNT of
// v_u c_u mod q for the T threads' elements of the tile (a few q, not reduced to
// [0, q): the split transform that follows takes values below 2^(k+3), the lazy
// one below 2^(k+5), the corrected one below 2q).  Sources come as two 30-bit halves (split_source), v = v0
// + v1 2^30, constants as two half-width limbs at 2^e, e = ceil(k/2), of c and
// c2 = 2^30 c mod q, so that the sum is A + B 2^e with two 64-bit sums of 32 x 32
// -> 64-bit products, four multiply-adds per term and no carries, and one
// reduction for all terms: 2^(2e) = rho mod q (delta or 2 delta) folds B's upper
// part, then a fold.  (A Shoup product and a correction per term, 23 instructions
// against 4, plus 9 per element.)  CNT = 1: c = 1, the source itself.  With vv
// (ModDown's exact lift), minus vP[vv[idx]] and h.  conv_split_ok has the bounds.
__device__ __forceinline__ uint64_t split_source(uint64_t v) {
  return (v & ((1u << 30) - 1)) | ((v >> 30) << 32);
}
__device__ __forceinline__ uint64_t join_source(uint64_t x) { return (x >> 32 << 30) | (uint32_t)x; }

template <int TILE, int T, int CNT>
__device__ __forceinline__ void conv_split_tile(uint64_t* sm, const uint64_t* wv, const uint64_t* w, const uint64_t* w2,
                                                uint32_t stride, const PrimeDev& pr, uint32_t tid,
                                                const uint32_t* vv = nullptr, const uint64_t* vP = nullptr,
                                                uint64_t h = 0) {
  const uint32_t e = (pr.k + 1) >> 1, mask = (1u << e) - 1, rho = pr.delta << (2 * e - pr.k);
  const uint64_t minus = 2 * pr.q - h;
  uint32_t c0[CNT], c1[CNT], d0[CNT], d1[CNT];
#pragma unroll
  for (int u = 0; u < CNT && CNT > 1; ++u) {
    const uint64_t x = w[(size_t)u * stride], y = w2[(size_t)u * stride];
    c0[u] = lo32(x) & mask;
    c1[u] = (uint32_t)(x >> e);
    d0[u] = lo32(y) & mask;
    d1[u] = (uint32_t)(y >> e);
  }
#pragma unroll 4
  for (uint32_t idx = tid; idx < (uint32_t)TILE; idx += T) {
    uint64_t a = 0, b = 0;
    if (CNT == 1) {
      a = wv[idx];
    } else {
#pragma unroll
      for (int u = 0; u < CNT; ++u) {
        const uint2 x = *reinterpret_cast<const uint2*>(wv + (size_t)u * TILE + idx);
        a = madw(x.x, c0[u], a);
        b = madw(x.x, c1[u], b);
        a = madw(x.y, d0[u], a);
        b = madw(x.y, d1[u], b);
      }
      a = madw(lo32(b) & mask, 1u << e, a);
      const uint64_t q = b >> e;  // below 2^35
      a = madw(lo32(q), rho, a);
      a = pack64(lo32(a), hi32(a) + hi32(q) * rho);
    }
    if (vv) a += minus - (CNT == 1 ? 0 : vP[vv[idx]]);
    sm[idx + (idx >> 3)] = fold(a, pr);
  }
}

// The same on T threads for a runtime count of 1 to 5 sources.
template <int TILE, int T>
__device__ __forceinline__ void conv_split(uint32_t cnt, uint64_t* sm, const uint64_t* wv, const uint64_t* w,
                                           const uint64_t* w2, uint32_t stride, const PrimeDev& pr, uint32_t tid,
                                           const uint32_t* vv = nullptr, const uint64_t* vP = nullptr, uint64_t h = 0) {
  if (cnt == 1) conv_split_tile<TILE, T, 1>(sm, wv, w, w2, stride, pr, tid, vv, vP, h);
  else if (cnt == 2) conv_split_tile<TILE, T, 2>(sm, wv, w, w2, stride, pr, tid, vv, vP, h);
  else if (cnt == 3) conv_split_tile<TILE, T, 3>(sm, wv, w, w2, stride, pr, tid, vv, vP, h);
  else if (cnt == 4) conv_split_tile<TILE, T, 4>(sm, wv, w, w2, stride, pr, tid, vv, vP, h);
  else conv_split_tile<TILE, T, 5>(sm, wv, w, w2, stride, pr, tid, vv, vP, h);
}

// The conversion of one tile for primes conv_split_ok turns down: Shoup
// products by the constants (w[u * stride], companions wsh), kept in [0, 2q),
// then to [0, q) and minus vP[vv[idx]] and h.  For the usual counts (CNT = 1 to
// 5) the constants sit in registers for the whole tile; CNT = 0 takes any cnt.
// (58-bit limbs, 61-bit special primes, N = 2^13, 64 rotations: ModUp 231 us with
// a runtime count beside the folded sums in one kernel, 193 with these in a kernel
// of their own; ModDown's conversion 190 and 159.)
template <int TILE, int T, int CNT>
__device__ __forceinline__ void conv_sum_tile(uint32_t cnt, uint64_t* sm, const uint64_t* wv, const uint64_t* w,
                                              const uint64_t* wsh, uint32_t stride, const PrimeDev& pr, uint32_t tid,
                                              const uint32_t* vv, const uint64_t* vP, uint64_t h) {
  const uint64_t q = pr.q, q2 = q + q;
  uint64_t cw[CNT ? CNT : 1], cs[CNT ? CNT : 1];
#pragma unroll
  for (int u = 0; u < CNT; ++u) {
    cw[u] = w[(size_t)u * stride];
    cs[u] = wsh[(size_t)u * stride];
  }
#pragma unroll 2
  for (uint32_t idx = tid; idx < (uint32_t)TILE; idx += T) {
    uint64_t y = 0;
    if (CNT) {
#pragma unroll
      for (int u = 0; u < CNT; ++u) {
        y += mul_shoup_lazy(wv[(size_t)u * TILE + idx], cw[u], cs[u], q);
        if (CNT > 1) y = y >= q2 ? y - q2 : y;
      }
    } else {
      for (uint32_t u = 0; u < cnt; ++u) {
        y += mul_shoup_lazy(wv[(size_t)u * TILE + idx], w[(size_t)u * stride], wsh[(size_t)u * stride], q);
        y = y >= q2 ? y - q2 : y;
      }
    }
    y = y >= q ? y - q : y;
    if (vv) y = sub_mod(sub_mod(y, vP[vv[idx]], q), h, q);
    sm[idx + (idx >> 3)] = y;
  }
}

template <int TILE, int T>
__device__ __forceinline__ void conv_sum(uint32_t cnt, uint64_t* sm, const uint64_t* wv, const uint64_t* w,
                                         const uint64_t* wsh, uint32_t stride, const PrimeDev& pr, uint32_t tid,
                                         const uint32_t* vv = nullptr, const uint64_t* vP = nullptr, uint64_t h = 0) {
  if (cnt == 1) conv_sum_tile<TILE, T, 1>(cnt, sm, wv, w, wsh, stride, pr, tid, vv, vP, h);
  else if (cnt == 2) conv_sum_tile<TILE, T, 2>(cnt, sm, wv, w, wsh, stride, pr, tid, vv, vP, h);
  else if (cnt == 3) conv_sum_tile<TILE, T, 3>(cnt, sm, wv, w, wsh, stride, pr, tid, vv, vP, h);
  else if (cnt == 4) conv_sum_tile<TILE, T, 4>(cnt, sm, wv, w, wsh, stride, pr, tid, vv, vP, h);
  else if (cnt == 5) conv_sum_tile<TILE, T, 5>(cnt, sm, wv, w, wsh, stride, pr, tid, vv, vP, h);
  else conv_sum_tile<TILE, T, 0>(cnt, sm, wv, w, wsh, stride, pr, tid, vv, vP, h);
}

// Column pass with the ModUp conversion in its load.  Grid: count * beta * nt * TILES.
template <int LOG_N, int LOG_M, int LOG_K>
__global__ void __launch_bounds__((1 << (LOG_M + LOG_K)) / 8) ks_modup_col(KsFusedArgs a) {
  using S = Shape<LOG_N, LOG_M, LOG_K, true>;
  constexpr uint32_t N = 1u << LOG_N;
  extern __shared__ __align__(16) unsigned char smem_raw[];
  ulonglong2* stw = reinterpret_cast<ulonglong2*>(smem_raw);
  uint64_t* sm = reinterpret_cast<uint64_t*>(smem_raw + sizeof(ulonglong2) * S::NTW);
  uint32_t b = blockIdx.x;
  const uint32_t tile = b % S::TILES;
  b /= S::TILES;
  const uint32_t t = b % a.nt;
  b /= a.nt;
  const uint32_t j = b % a.beta, i = b / a.beta;
  const uint32_t lo = a.lo[j], cnt = a.cnt[j];
  if (t >= lo && t < lo + cnt) {  // the digit's own limbs are used as they are
    pdl_wait();
    return;
  }
  const uint32_t prime = ks_prime(t, a.level, a.L);
  const PrimeDev pr = a.primes[prime];
  stage_twiddles<LOG_N, LOG_M, LOG_K, true>(stw, a.tw + (size_t)prime * N, tile);
  pdl_wait();
  const uint64_t* tab = a.consts + a.off[j];
  const uint64_t* mat = tab + 2 * cnt;
  const uint64_t* mat_sh = mat + (size_t)cnt * a.np;
  const uint64_t* x = a.d2c + (size_t)i * a.level * N;
  const uint64_t q2 = pr.q + pr.q;
#pragma unroll 2
  for (uint32_t idx = threadIdx.x; idx < (uint32_t)S::TILE; idx += S::T) {
    const uint32_t xx = idx >> LOG_K, k = idx & (S::K - 1);
    const uint32_t e = S::gidx(tile, k, xx);
    uint64_t y;
    if (cnt == 1) {
      y = reduce64(x[(size_t)lo * N + e], pr);  // Q_j / q_lo = 1
    } else {
      // products by the constant (Q_j/q_i) mod q_t are Shoup products in [0, 2q), kept in [0, 2q)
      y = 0;
      for (uint32_t u = 0; u < cnt; ++u) {
        const uint64_t qa = a.primes[lo + u].q;
        const uint64_t v = mul_shoup(x[(size_t)(lo + u) * N + e], tab[2 * u], tab[2 * u + 1], qa);
        y += mul_shoup_lazy(v, mat[(size_t)u * a.np + prime], mat_sh[(size_t)u * a.np + prime], pr.q);
        y = y >= q2 ? y - q2 : y;
      }
      y = y >= pr.q ? y - pr.q : y;
    }
    sm[idx + (idx >> 3)] = y;
  }
  __syncthreads();
  uint64_t* out = a.ext + (((size_t)i * a.beta + j) * a.nt + t) * N;
  run_rounds<false, LOG_N, LOG_M, LOG_K, true>(sm, stw, pr, threadIdx.x);
#pragma unroll 8
  for (uint32_t idx = threadIdx.x; idx < (uint32_t)S::TILE; idx += S::T) {
    const uint32_t xx = idx >> LOG_K, k = idx & (S::K - 1);
    out[S::gidx(tile, k, xx)] = sm[idx + (idx >> 3)];
  }
}

// The same column pass for several target limbs of one digit and tile in one
// CTA: the digit's limbs are read once and their products by
// (Q_j/q_i)^-1 mod q_i (or, for a one-limb digit, the limb itself) are kept
// in shared memory for those targets.  The nt targets are shared evenly by
// a.splits CTAs, and by the G groups of T threads of a CTA, each with its own
// tile and twiddles (the sources' tiles are what limits the CTAs of an SM, so
// groups are how its warps are filled; conv_plan).  SPLIT: every target's
// conversion runs as conv_split_tile (else all as conv_sum; an instance each, as
// the two in one kernel cost both registers).  Grid: count * beta * splits
// * TILES; dynamic shared memory: [G] twiddles, [G] tiles, cnt_max * TILE words.
template <int LOG_N, int LOG_M, int LOG_K, int G, bool SPLIT>
__global__ void __launch_bounds__(G * ((1 << (LOG_M + LOG_K)) / 8), 1024 / (G * ((1 << (LOG_M + LOG_K)) / 8)))
ks_modup_col_all(KsFusedArgs a) {
  using S = Shape<LOG_N, LOG_M, LOG_K, true>;
  constexpr uint32_t N = 1u << LOG_N, TW = S::TILE + S::TILE / 8;
  extern __shared__ __align__(16) unsigned char smem_raw[];
  const uint32_t grp = G == 1 ? 0u : threadIdx.x / S::T, tid = G == 1 ? threadIdx.x : threadIdx.x % S::T;
  ulonglong2* stw = reinterpret_cast<ulonglong2*>(smem_raw) + grp * S::NTW;
  uint64_t* sm0 = reinterpret_cast<uint64_t*>(smem_raw + sizeof(ulonglong2) * S::NTW * G);
  uint64_t* sm = sm0 + grp * TW;
  uint64_t* wv = sm0 + G * TW;  // [cnt][TILE]
  uint32_t b = blockIdx.x;
  const uint32_t tile = b % S::TILES;
  b /= S::TILES;
  const uint32_t part = b % a.splits;
  b /= a.splits;
  const uint32_t j = b % a.beta, i = b / a.beta;
  const uint32_t lo = a.lo[j], cnt = a.cnt[j];
  const uint32_t t_end = (part + 1) * a.nt / a.splits;
  const uint64_t* tab = a.consts + a.off[j];
  const uint64_t* mat = tab + 2 * cnt;
  const uint64_t* mat_sh = mat + (size_t)cnt * a.np;
  const uint64_t* mat_2 = mat_sh + (size_t)cnt * a.np + 2 * cnt;
  const uint64_t* x = a.d2c + (size_t)i * a.level * N;
  const bool halves = SPLIT && cnt > 1;
  for (uint32_t u = grp; u < cnt; u += G) {
    const PrimeDev pa = a.primes[lo + u];
    if (a.half) {
      // the inverse transform's column pass on this tile, then the scaling by
      // N^-1 and the product by (Q_j/q_i)^-1 as one constant
      stage_twiddles<LOG_N, LOG_M, LOG_K, true>(stw, a.itw + (size_t)(lo + u) * N, tile, tid, S::T);
      pdl_wait();
#pragma unroll 8
      for (uint32_t idx = tid; idx < (uint32_t)S::TILE; idx += S::T) {
        const uint32_t e = S::gidx(tile, idx & (S::K - 1), idx >> LOG_K);
        sm[idx + (idx >> 3)] = x[(size_t)(lo + u) * N + e];
      }
      group_sync<G, S::T>(grp);
      run_rounds<true, LOG_N, LOG_M, LOG_K, true, 3, G>(sm, stw, pa, tid, grp);
      const uint64_t* tabn = mat_sh + (size_t)cnt * a.np;
      const uint64_t w = tabn[2 * u], wsh = tabn[2 * u + 1];
#pragma unroll 8
      for (uint32_t idx = tid; idx < (uint32_t)S::TILE; idx += S::T) {
        const uint64_t v = mul_shoup(sm[idx + (idx >> 3)], w, wsh, pa.q);
        wv[(size_t)u * S::TILE + idx] = halves ? split_source(v) : v;
      }
    } else {
      pdl_wait();
#pragma unroll 8
      for (uint32_t idx = tid; idx < (uint32_t)S::TILE; idx += S::T) {
        const uint32_t e = S::gidx(tile, idx & (S::K - 1), idx >> LOG_K);
        const uint64_t xv = x[(size_t)(lo + u) * N + e];
        const uint64_t v = cnt == 1 ? xv : mul_shoup(xv, tab[2 * u], tab[2 * u + 1], pa.q);
        wv[(size_t)u * S::TILE + idx] = halves ? split_source(v) : v;
      }
    }
    // the next limb's staging overwrites stw and sm: wait for every thread
    group_sync<G, S::T>(grp);
  }
  pdl_wait();  // (groups without a source)
  if (G > 1) __syncthreads();  // every group's sources
  for (uint32_t t = part * a.nt / a.splits + grp; t < t_end; t += G) {
    if (t >= lo && t < lo + cnt) continue;  // the digit's own limbs are used as they are
    const uint32_t prime = ks_prime(t, a.level, a.L);
    const PrimeDev pr = a.primes[prime];
    // the previous target's rounds ended with a barrier, and its write-out
    // reads only the words each thread rewrites below
    stage_twiddles<LOG_N, LOG_M, LOG_K, true>(stw, a.tw + (size_t)prime * N, tile, tid, S::T);
    if (SPLIT) conv_split<S::TILE, S::T>(cnt, sm, wv, mat + prime, mat_2 + prime, a.np, pr, tid);
    else conv_sum<S::TILE, S::T>(cnt, sm, wv, mat + prime, mat_sh + prime, a.np, pr, tid);
    group_sync<G, S::T>(grp);
    uint64_t* out = a.ext + (((size_t)i * a.beta + j) * a.nt + t) * N;
    run_rounds<false, LOG_N, LOG_M, LOG_K, true, 3, G>(sm, stw, pr, tid, grp);
#pragma unroll 8
    for (uint32_t idx = tid; idx < (uint32_t)S::TILE; idx += S::T) {
      const uint32_t xx = idx >> LOG_K, k = idx & (S::K - 1);
      out[S::gidx(tile, k, xx)] = sm[idx + (idx >> 3)];
    }
  }
}

// ---- hoisted rotate-and-sum ------------------------------------------------
// The rotations of one rotate-and-sum stage share the decomposition of the
// input: the column pass (ks_modup_col[_all], run once) and the row pass of
// every digit.  Rotation r then needs the products of the permuted digits,
//   acc_r[e] = sum_j D_j[src_r(e)] * evk_r[j][e],  src_r = automorph_src(., gal_r),
// with a permutation of the evaluation points that maps rows to rows: in
// bit-reversed order a row of M points is a residue class of the natural
// index modulo N/M, and X -> X^gal maps residue classes onto residue
// classes.  When every rotation maps each CTA's rows onto themselves (a
// closed stage), ks_row_rot runs the row pass and sums all rotations for its
// own positions from the tiles it holds in shared memory; otherwise the row
// pass runs by itself and ks_gather_rot fetches the rows each rotation reads.
static_assert(HE_MAX_ROT * HE_MAX_PRIMES <= kSplit3Terms, "products of a stage (rotations times digits)");
struct KsRotArgs {
  KsFusedArgs k;           // k.acc: the accumulator (summed over the rotations)
  uint32_t nrot, count;
  int reduce_each;         // nrot * beta products could exceed 128 bits: reduce after each rotation
  uint64_t gal[HE_MAX_ROT];
  const uint64_t* evk[HE_MAX_ROT];
  // part 0 of the input (evaluation form, count x [level][N] at c0_stride):
  // when set, part 0 of the accumulator's limbs q_t also receives
  // (P mod q_t) * sum_r kappa_r(c0), which the ModDown turns into
  // sum_r kappa_r(c0) exactly (nullptr: not added; in ks_row_rot only where
  // the target limbs q_t all take the split sums)
  const uint64_t* c0;
  uint64_t c0_stride;
  // the merged ModDown's dropped limb (pd_limb: that limb, or beyond the targets):
  // acc there also receives P d, both parts (pd_w: P mod q, Shoup pair).  Only in
  // the key switch's kernel of small grids (ks_row_rot with digit groups), where
  // launches count; the registers it takes cost ks_row_rot's others 3 %, more than
  // the separate kernel.
  CtBatch pd;
  uint32_t pd_limb;
  uint64_t pd_w, pd_wsh;
};

// The residue of a split sum, with part 0's term s0 pm (s0 a sum of up to 16
// residues, pm = P mod q) when add.
__device__ __forceinline__ uint64_t split3_final(uint64_t ll, uint64_t hh, uint64_t ss, uint32_t sb, const PrimeDev& pr,
                                                 bool add, uint64_t s0, uint64_t pm) {
  if (pr.delta) {
    if (add) {
      const uint32_t mask = (1u << sb) - 1;
      mac_split3(ll, hh, ss, split3(fold(s0, pr), sb, mask), split3(pm, sb, mask));
    }
    return split3_residue(ll, hh, ss, sb, pr);
  }
  uint64_t lo, hi;
  split3_total(ll, hh, ss, sb, lo, hi);
  if (add) mac128(lo, hi, s0, pm);
  return reduce128_any(hi, lo, pr);
}

// Grid: nt * ceil(count / CT) * TILES, target limb slowest and row tile
// fastest, so that the CTAs resident at one time share their keys (one limb
// of each rotation's key) in L2 and finish each ciphertext's limb together.
// A CTA holds CT ciphertexts of one limb and tile: group g of T threads runs
// the row passes of ciphertext i0 + g, and in a closed stage every thread
// then sums the products for its positions of all CT ciphertexts, so each
// key word it loads serves CT ciphertexts (8/CT bytes of key per key
// product).  CT > 1 only for closed stages; a tail CTA repeats its last
// ciphertext in the groups beyond the count and stores nothing for them.
// In small grids (DG > 1, CT = 1) DG groups share one ciphertext's digits: each
// runs the row pass of every DG-th digit, so the passes run side by side instead
// of in pairs one after the other, and all threads sum the products.
// Shared memory: the tile's twiddles, every digit's transformed tile of each
// ciphertext ([CT][beta][TILE + TILE/8] words) and, with ra.c0, each
// ciphertext's part-0 tile ([CT][TILE + TILE/8]).
template <int LOG_N, int LOG_M, int LOG_K, int CT, int DG>
__global__ void __launch_bounds__(CT * DG * ((1 << (LOG_M + LOG_K)) / 8), DG > 1 ? 1 : 4 / CT) ks_row_rot(KsRotArgs ra) {
  using S = Shape<LOG_N, LOG_M, LOG_K, false>;
  constexpr uint32_t N = 1u << LOG_N;
  constexpr int PER = S::TILE / S::T;  // 8
  constexpr uint32_t TW = S::TILE + S::TILE / 8;
  static_assert((CT == 1 || CT == 2 || CT == 4) && (DG == 1 || CT == 1), "ciphertexts and digit groups per CTA");
  const KsFusedArgs& a = ra.k;
  extern __shared__ __align__(16) unsigned char smem_raw[];
  ulonglong2* stw = reinterpret_cast<ulonglong2*>(smem_raw);
  uint64_t* dig = reinterpret_cast<uint64_t*>(smem_raw + sizeof(ulonglong2) * S::NTW);
  uint32_t b = blockIdx.x;
  const uint32_t tile = b % S::TILES;
  b /= S::TILES;
  const uint32_t ngrp = (ra.count + CT - 1) / CT;
  const uint32_t i0 = (b % ngrp) * CT, t = b / ngrp;
  constexpr uint32_t NG = CT * DG;                                   // groups of T threads
  const uint32_t gid = NG == 1 ? 0u : threadIdx.x / S::T;            // warp-uniform: T is a multiple of 32
  const uint32_t ltid = NG == 1 ? threadIdx.x : threadIdx.x % S::T;
  const uint32_t grp = gid / DG, dg = gid % DG;                      // ciphertext, digit group
  const uint32_t i = min(i0 + grp, ra.count - 1);
  const uint32_t prime = ks_prime(t, a.level, a.L);
  const PrimeDev pr = a.primes[prime];
  const uint64_t q = pr.q;
  // the input's part 0, added through each rotation on the limbs q_t
  const bool add_c0 = ra.c0 && t < a.level;
  uint64_t* c0s = dig + (size_t)CT * a.beta * TW;  // its tiles, [CT][TW] after every digit tile
  // 1. every digit's tile in evaluation form, canonical residues: the
  // twiddles and all digit tiles are copied asynchronously up front (one
  // group each, part 0's tile with the last), so that later tiles arrive
  // while earlier ones transform
  stage_twiddles_async<LOG_N, LOG_M, LOG_K, false>(stw, a.tw + (size_t)prime * N, tile, threadIdx.x, NG * S::T);
  cp_async_commit();
  pdl_wait();
  for (uint32_t j = dg; j < a.beta; j += DG) {
    uint64_t* sm = dig + ((size_t)grp * a.beta + j) * TW;
    const bool own = t >= a.lo[j] && t < a.lo[j] + a.cnt[j];
    const uint64_t* src = own ? a.d + (size_t)i * a.d_stride + (size_t)t * N
                              : a.ext + (((size_t)i * a.beta + j) * a.nt + t) * N;
    // the own limb is read through the input's automorphism (a single
    // rotation's key switch: the converted tiles already are)
    const uint64_t in_gal = own ? a.gal : 0;
#pragma unroll
    for (int u = 0; u < PER; ++u) {
      const uint32_t idx = ltid + u * S::T;
      const uint32_t e = S::gidx(tile, idx >> LOG_M, idx & (S::M - 1));
      cp_async8(sm + idx + (idx >> 3), src + (in_gal ? automorph_src(e, in_gal, LOG_N) : e));
    }
    if (add_c0 && j + 1 == a.beta) {
      const uint64_t* s0 = ra.c0 + (size_t)i * ra.c0_stride + (size_t)t * N;
#pragma unroll
      for (int u = 0; u < PER; ++u) {
        const uint32_t idx = ltid + u * S::T;
        cp_async8(c0s + (size_t)grp * TW + idx + (idx >> 3), s0 + S::gidx(tile, idx >> LOG_M, idx & (S::M - 1)));
      }
    }
    cp_async_commit();
  }
  // the converted digits' row passes, two tiles at a time (one barrier per
  // round for both, each twiddle loaded once for both)
  auto finish_tile = [&](uint64_t* sm) {
#pragma unroll
    for (int u = 0; u < PER; ++u) {
      const uint32_t idx = ltid + u * S::T;
      const uint64_t v = sm[idx + (idx >> 3)];
      sm[idx + (idx >> 3)] = fwd_final(v, pr);
    }
  };
  if constexpr (DG > 1) {
    cp_async_wait<0>();
    __syncthreads();  // the twiddles, which all threads copied
    for (uint32_t j = dg; j < a.beta; j += DG) {
      if (t >= a.lo[j] && t < a.lo[j] + a.cnt[j]) continue;
      uint64_t* sm = dig + (size_t)j * TW;
      run_rounds<false, LOG_N, LOG_M, LOG_K, false, 3, DG>(sm, stw, pr, ltid, dg);
      finish_tile(sm);
    }
  } else {
    int pend = -1;  // a converted digit waiting for a partner
    for (uint32_t j = 0; j < a.beta; ++j) {
      const bool own = t >= a.lo[j] && t < a.lo[j] + a.cnt[j];
      if (own) continue;
      if (pend < 0) {
        pend = (int)j;
        continue;
      }
      cp_async_wait_dyn(a.beta - 1 - j);  // the twiddles and tiles 0 .. j have arrived
      __syncthreads();
      uint64_t* sms[2] = {dig + ((size_t)grp * a.beta + (uint32_t)pend) * TW, dig + ((size_t)grp * a.beta + j) * TW};
      run_rounds_n<false, LOG_N, LOG_M, LOG_K, false, 2>(sms, stw, pr, ltid);
      finish_tile(sms[0]);
      finish_tile(sms[1]);
      pend = -1;
    }
    if (pend >= 0) {
      uint64_t* sm = dig + ((size_t)grp * a.beta + (uint32_t)pend) * TW;
      cp_async_wait_dyn(a.beta - 1 - (uint32_t)pend);
      __syncthreads();
      run_rounds<false, LOG_N, LOG_M, LOG_K, false>(sm, stw, pr, ltid);
      finish_tile(sm);
    }
  }
  cp_async_wait<0>();  // the own limb's tile
  __syncthreads();
  // 2. the products of the permuted digits with each rotation's key, summed
  // exactly (split sums or 128-bit sums) and reduced once per residue
  const uint32_t row0 = (uint32_t)tile << LOG_K;
  auto add_pd = [&](uint32_t ct, uint32_t p, uint32_t e, uint64_t v) {
    return add_mod(v, mul_shoup(cpoly(ra.pd, ct, p, t, N)[e], ra.pd_w, ra.pd_wsh, q), q);
  };
  // key products as split sums (mac_split3) when the prime and the number of
  // summed terms allow it
  const uint32_t sb = (pr.k + 1) >> 1;
  if (split3_fits(pr.k, ra.nrot * a.beta)) {
    // one pair of neighbouring positions per pass, all CT ciphertexts with
    // each key load
    constexpr int PPT = PER / 2 / NG;
    const uint32_t mask = (1u << sb) - 1;
    uint64_t pm = 1;  // P mod q_t
    if (add_c0)
      for (uint32_t u = 0; u < a.alpha; ++u) pm = mul_mod(pm, reduce64(a.primes[a.L + u].q, pr), pr);
#pragma unroll 1
    for (int v0 = 0; v0 < PPT; ++v0) {
      const uint32_t idx = 2 * (threadIdx.x + v0 * NG * S::T);
      const uint32_t eo = S::gidx(tile, idx >> LOG_M, idx & (S::M - 1));
      uint64_t ll[CT][2][2], hh[CT][2][2], ss[CT][2][2];  // [ciphertext][part][position]
      uint64_t s0[CT][2];                                  // sum_r kappa_r(c0) (below nrot q)
#pragma unroll
      for (int c = 0; c < CT; ++c) {
        s0[c][0] = s0[c][1] = 0;
#pragma unroll
        for (int p = 0; p < 2; ++p)
#pragma unroll
          for (int u = 0; u < 2; ++u) ll[c][p][u] = hh[c][p][u] = ss[c][p][u] = 0;
      }
      for (uint32_t r = 0; r < ra.nrot; ++r) {
        uint32_t so[2];
#pragma unroll
        for (int u = 0; u < 2; ++u) {
          const uint32_t p = automorph_src(eo + u, ra.gal[r], LOG_N);
          const uint32_t sl = (((p >> LOG_M) - row0) << LOG_M) | (p & (S::M - 1));
          so[u] = sl + (sl >> 3);
        }
        if (add_c0)
#pragma unroll
          for (int c = 0; c < CT; ++c) {
            s0[c][0] += c0s[(size_t)c * TW + so[0]];
            s0[c][1] += c0s[(size_t)c * TW + so[1]];
          }
        const uint64_t* ev = ra.evk[r];
#pragma unroll 2
        for (uint32_t j = 0; j < a.beta; ++j) {
          const uint64_t* kb = ev + (((size_t)j * 2 + 0) * a.np + prime) * N;
          const uint64_t* ka = ev + (((size_t)j * 2 + 1) * a.np + prime) * N;
          const ulonglong2 wb = __ldg(reinterpret_cast<const ulonglong2*>(kb + eo));
          const ulonglong2 wa = __ldg(reinterpret_cast<const ulonglong2*>(ka + eo));
          const Split3 kb0 = split3(wb.x, sb, mask), kb1 = split3(wb.y, sb, mask);
          const Split3 ka0 = split3(wa.x, sb, mask), ka1 = split3(wa.y, sb, mask);
#pragma unroll
          for (int c = 0; c < CT; ++c) {
            const uint64_t* sm = dig + ((size_t)c * a.beta + j) * TW;
            const Split3 x0 = split3(sm[so[0]], sb, mask), x1 = split3(sm[so[1]], sb, mask);
            mac_split3(ll[c][0][0], hh[c][0][0], ss[c][0][0], x0, kb0);
            mac_split3(ll[c][0][1], hh[c][0][1], ss[c][0][1], x1, kb1);
            mac_split3(ll[c][1][0], hh[c][1][0], ss[c][1][0], x0, ka0);
            mac_split3(ll[c][1][1], hh[c][1][1], ss[c][1][1], x1, ka1);
          }
        }
      }
#pragma unroll
      for (int c = 0; c < CT; ++c) {
        if (i0 + c >= ra.count) break;
        uint64_t* o0 = a.acc + ((size_t)(i0 + c) * 2 * a.nt + t) * N;
#pragma unroll
        for (int p = 0; p < 2; ++p) {
          uint64_t r2[2];
#pragma unroll
          for (int u = 0; u < 2; ++u) {
            r2[u] = split3_final(ll[c][p][u], hh[c][p][u], ss[c][p][u], sb, pr, p == 0 && add_c0, s0[c][u], pm);
            if (DG > 1 && t == ra.pd_limb) r2[u] = add_pd(i0 + c, p, eo + u, r2[u]);
          }
          *reinterpret_cast<ulonglong2*>(o0 + (size_t)p * a.nt * N + eo) = make_ulonglong2(r2[0], r2[1]);
        }
      }
    }
    return;
  }
  {
    // each thread sums every rotation's products for its own positions, two
    // neighbouring positions at a time (16-byte key loads and stores), for
    // all CT ciphertexts with each key load
    constexpr int PPT = PER / 2 / NG;          // position pairs per thread
    constexpr int PAIRS = PPT < 2 ? PPT : 2;   // pairs per pass (bounds the registers)
    constexpr int NP = 2 * PAIRS;              // positions per pass
#pragma unroll 1
    for (int v0 = 0; v0 < PPT; v0 += PAIRS) {
      uint32_t eo[PAIRS];  // first of the two positions (even)
      uint64_t a0l[CT][NP], a0h[CT][NP], a1l[CT][NP], a1h[CT][NP];  // 128-bit sums of full products
#pragma unroll
      for (int v = 0; v < PAIRS; ++v) {
        const uint32_t idx = 2 * (threadIdx.x + (v0 + v) * NG * S::T);
        eo[v] = S::gidx(tile, idx >> LOG_M, idx & (S::M - 1));
      }
#pragma unroll
      for (int c = 0; c < CT; ++c)
#pragma unroll
        for (int u = 0; u < NP; ++u) a0l[c][u] = a0h[c][u] = a1l[c][u] = a1h[c][u] = 0;
      for (uint32_t r = 0; r < ra.nrot; ++r) {
        uint32_t so[NP];
#pragma unroll
        for (int u = 0; u < NP; ++u) {
          const uint32_t p = automorph_src(eo[u >> 1] + (u & 1), ra.gal[r], LOG_N);
          const uint32_t sl = (((p >> LOG_M) - row0) << LOG_M) | (p & (S::M - 1));
          so[u] = sl + (sl >> 3);
        }
        const uint64_t* ev = ra.evk[r];
#pragma unroll 2
        for (uint32_t j = 0; j < a.beta; ++j) {
          const uint64_t* kb = ev + (((size_t)j * 2 + 0) * a.np + prime) * N;
          const uint64_t* ka = ev + (((size_t)j * 2 + 1) * a.np + prime) * N;
#pragma unroll
          for (int v = 0; v < PAIRS; ++v) {
            const ulonglong2 wb = __ldg(reinterpret_cast<const ulonglong2*>(kb + eo[v]));
            const ulonglong2 wa = __ldg(reinterpret_cast<const ulonglong2*>(ka + eo[v]));
#pragma unroll
            for (int c = 0; c < CT; ++c) {
              const uint64_t* sm = dig + ((size_t)c * a.beta + j) * TW;
              const uint64_t x0 = sm[so[2 * v]], x1 = sm[so[2 * v + 1]];
              mac128(a0l[c][2 * v], a0h[c][2 * v], x0, wb.x);
              mac128(a0l[c][2 * v + 1], a0h[c][2 * v + 1], x1, wb.y);
              mac128(a1l[c][2 * v], a1h[c][2 * v], x0, wa.x);
              mac128(a1l[c][2 * v + 1], a1h[c][2 * v + 1], x1, wa.y);
            }
          }
        }
      }
#pragma unroll
      for (int c = 0; c < CT; ++c) {
        if (i0 + c >= ra.count) break;
        uint64_t* o0 = a.acc + ((size_t)(i0 + c) * 2 * a.nt + t) * N;
        uint64_t* o1 = o0 + (size_t)a.nt * N;
#pragma unroll
        for (int v = 0; v < PAIRS; ++v) {
          uint64_t r2[2][2];
#pragma unroll
          for (int u = 0; u < 2; ++u) {
            r2[0][u] = reduce128_any(a0h[c][2 * v + u], a0l[c][2 * v + u], pr);
            r2[1][u] = reduce128_any(a1h[c][2 * v + u], a1l[c][2 * v + u], pr);
            if (DG > 1 && t == ra.pd_limb)
              for (uint32_t p = 0; p < 2; ++p) r2[p][u] = add_pd(i0 + c, p, eo[v] + u, r2[p][u]);
          }
          *reinterpret_cast<ulonglong2*>(o0 + eo[v]) = make_ulonglong2(r2[0][0], r2[0][1]);
          *reinterpret_cast<ulonglong2*>(o1 + eo[v]) = make_ulonglong2(r2[1][0], r2[1][1]);
        }
      }
    }
  }
}

// Stages with rotations that move rows between tiles: the row pass runs
// by itself (ntt2's, in place on the column pass's outputs) and this kernel
// gathers.  A CTA of target limb t owns one block of output positions and CT
// ciphertexts.  Step (r, j) needs the words of digit j that rotation r moves to
// the block (any aligned block of 2^k positions is a residue class like a row,
// so they are one block too) of each ciphertext and the key's two
// polynomials at the block; a ring of kGatherRing steps is kept in flight with
// cp.async, since a step computes for about 0.3 us and its key words come from
// HBM.  A thread sums one pair of neighbouring positions, like the closed
// stages; each accumulator residue is reduced and written once.  Part 0 (ra.c0)
// is one more step per rotation.  Bound by its instructions (FMA pipe 53 %,
// issue slots half used, DRAM 28 %).  Fifteen unit steps at N = 2^16, 24 limbs,
// four ciphertexts: 1.44 ms (1.68 with one CTA of 1024 positions per SM instead
// of two of 512), and 0.34 ms for the row pass (every rotation's
// reduced products added to the rows they move to with 64-bit atomics: 2.84 ms;
// a rotation's digits per step and keys read by the products: 2.79 ms).
// Grid: nt * ceil(count / CT) * N / BLK, blocks of one limb's neighbouring CTAs
// sharing its key words in L2.
constexpr int kGatherThreads = 256, kGatherRing = 6;

template <int LOG_N, int CT>
__global__ void __launch_bounds__(kGatherThreads, 2) ks_gather_rot(KsRotArgs ra) {
  constexpr uint32_t N = 1u << LOG_N, BLK = 2 * kGatherThreads, SLOT = (CT + 2) * BLK;
  const KsFusedArgs& a = ra.k;
  extern __shared__ __align__(16) unsigned char smem_raw[];
  uint64_t* buf = reinterpret_cast<uint64_t*>(smem_raw);  // [ring][CT digit blocks, key b, key a][BLK]
  uint32_t b = blockIdx.x;
  const uint32_t blk = b % (N / BLK);
  b /= N / BLK;
  const uint32_t ngrp = (ra.count + CT - 1) / CT;
  const uint32_t i0 = (b % ngrp) * CT, t = b / ngrp;
  const uint32_t prime = ks_prime(t, a.level, a.L);
  const PrimeDev pr = a.primes[prime];
  const bool add_c0 = ra.c0 && t < a.level;
  const uint32_t ntile = a.beta + (add_c0 ? 1 : 0), nsteps = ra.nrot * ntile;
  const uint32_t idx = 2 * threadIdx.x, eo = blk * BLK + idx;
  // where digit j's row starts: the digit's converted limb (one digit is nt
  // limbs apart from the next), the input's own limb in digit jo, part 0
  const uint64_t *ext[CT], *own[CT], *c0[CT];
#pragma unroll
  for (int c = 0; c < CT; ++c) {
    const uint32_t i = min(i0 + c, ra.count - 1);
    ext[c] = a.ext + ((size_t)i * a.beta * a.nt + t) * N;
    own[c] = a.d + (size_t)i * a.d_stride + (size_t)t * N;
    c0[c] = add_c0 ? ra.c0 + (size_t)i * ra.c0_stride + (size_t)t * N : nullptr;
  }
  const uint32_t to0 = (uint32_t)__cvta_generic_to_shared(buf + idx);
  uint32_t jo = a.beta;  // (none)
  for (uint32_t j = 0; j < a.beta; ++j)
    if (t >= a.lo[j] && t < a.lo[j] + a.cnt[j]) jo = j;
  const uint32_t ext_step = a.nt * N, key_step = a.np * N;  // 2 beta np N < 2^32
  uint32_t cr = 0, cj = 0;  // the next step to copy
  uint32_t off = 0, ko = 0, eoff = 0;
  const uint64_t* key = nullptr;
  auto next_rotation = [&]() {
    off = (automorph_src(blk * BLK, ra.gal[cr], LOG_N) & ~(BLK - 1)) | idx;
    key = ra.evk[cr];
    ko = prime * N + eo;
    eoff = off;
  };
  next_rotation();
  auto copy_step = [&](uint32_t slot) {
    if (cr < ra.nrot) {
      const uint32_t to = to0 + 8 * slot * SLOT;
      if (cj < a.beta) {
        if (cj == jo)
#pragma unroll
          for (int c = 0; c < CT; ++c) cp_async16_s(to + 8 * c * BLK, own[c] + off);
        else
#pragma unroll
          for (int c = 0; c < CT; ++c) cp_async16_s(to + 8 * c * BLK, ext[c] + eoff);
        cp_async16_s(to + 8 * CT * BLK, key + ko);
        cp_async16_s(to + 8 * (CT + 1) * BLK, key + (ko + key_step));
        ko += 2 * key_step;
        eoff += ext_step;
      } else {
#pragma unroll
        for (int c = 0; c < CT; ++c) cp_async16_s(to + 8 * c * BLK, c0[c] + off);
      }
      if (++cj == ntile) {
        cj = 0;
        if (++cr < ra.nrot) next_rotation();
      }
    }
    cp_async_commit();  // (an empty group past the last step keeps the count)
  };
  const uint32_t sb = (pr.k + 1) >> 1, mask = (1u << (sb & 31)) - 1;
  const bool split = split3_fits(pr.k, ra.nrot * a.beta);
  // split sums (ll, hh, ss), or 128-bit sums (ll = low word, hh = high word)
  uint64_t ll[CT][2][2], hh[CT][2][2], ss[CT][2][2], s0[CT][2];  // [ciphertext][part][position]
#pragma unroll
  for (int c = 0; c < CT; ++c) {
    s0[c][0] = s0[c][1] = 0;
#pragma unroll
    for (int p = 0; p < 2; ++p)
#pragma unroll
      for (int u = 0; u < 2; ++u) ll[c][p][u] = hh[c][p][u] = ss[c][p][u] = 0;
  }
  pdl_wait();
#pragma unroll 1
  for (uint32_t s = 0; s < kGatherRing - 1; ++s) copy_step(s);
  uint32_t slot = 0;
  for (uint32_t r = 0; r < ra.nrot; ++r) {
    // the sources of two neighbouring positions are neighbours (their exponents
    // differ by N, and gal is odd): one 16-byte load, its words swapped or not
    const uint32_t sp0 = automorph_src(eo, ra.gal[r], LOG_N) & (BLK - 1);
    const uint32_t sp = sp0 & ~1u;
    const bool sw = sp0 & 1;
    for (uint32_t j = 0; j < ntile; ++j) {
      cp_async_wait<kGatherRing - 2>();  // this step's group has arrived
      __syncthreads();                   // for every thread; and the slot before it is free
      copy_step(slot == 0 ? kGatherRing - 1 : slot - 1);
      const uint64_t* sm = buf + slot * SLOT;
      slot = slot + 1 == kGatherRing ? 0 : slot + 1;
      if (j == a.beta) {
#pragma unroll
        for (int c = 0; c < CT; ++c) {
          const ulonglong2 xv = *reinterpret_cast<const ulonglong2*>(sm + c * BLK + sp);
          s0[c][0] += sw ? xv.y : xv.x;
          s0[c][1] += sw ? xv.x : xv.y;
        }
        continue;
      }
      const ulonglong2 wb = *reinterpret_cast<const ulonglong2*>(sm + CT * BLK + idx);
      const ulonglong2 wa = *reinterpret_cast<const ulonglong2*>(sm + (CT + 1) * BLK + idx);
      if (split) {
        const Split3 kb0 = split3(wb.x, sb, mask), kb1 = split3(wb.y, sb, mask);
        const Split3 ka0 = split3(wa.x, sb, mask), ka1 = split3(wa.y, sb, mask);
#pragma unroll
        for (int c = 0; c < CT; ++c) {
          const ulonglong2 xv = *reinterpret_cast<const ulonglong2*>(sm + c * BLK + sp);
          const Split3 x0 = split3(sw ? xv.y : xv.x, sb, mask), x1 = split3(sw ? xv.x : xv.y, sb, mask);
          mac_split3(ll[c][0][0], hh[c][0][0], ss[c][0][0], x0, kb0);
          mac_split3(ll[c][0][1], hh[c][0][1], ss[c][0][1], x1, kb1);
          mac_split3(ll[c][1][0], hh[c][1][0], ss[c][1][0], x0, ka0);
          mac_split3(ll[c][1][1], hh[c][1][1], ss[c][1][1], x1, ka1);
        }
      } else {
#pragma unroll
        for (int c = 0; c < CT; ++c) {
          const ulonglong2 xv = *reinterpret_cast<const ulonglong2*>(sm + c * BLK + sp);
          const uint64_t x0 = sw ? xv.y : xv.x, x1 = sw ? xv.x : xv.y;
          mac128(ll[c][0][0], hh[c][0][0], x0, wb.x);
          mac128(ll[c][0][1], hh[c][0][1], x1, wb.y);
          mac128(ll[c][1][0], hh[c][1][0], x0, wa.x);
          mac128(ll[c][1][1], hh[c][1][1], x1, wa.y);
        }
      }
    }
    if (!split && ra.reduce_each)  // nrot * beta products could leave 128 bits: beta at a time
#pragma unroll
      for (int c = 0; c < CT; ++c)
#pragma unroll
        for (int p = 0; p < 2; ++p)
#pragma unroll
          for (int u = 0; u < 2; ++u) {
            ll[c][p][u] = reduce128_any(hh[c][p][u], ll[c][p][u], pr);
            hh[c][p][u] = 0;
          }
  }
  uint64_t pm = 1;  // P mod q_t
  if (add_c0)
    for (uint32_t u = 0; u < a.alpha; ++u) pm = mul_mod(pm, reduce64(a.primes[a.L + u].q, pr), pr);
#pragma unroll
  for (int c = 0; c < CT; ++c) {
    if (i0 + c >= ra.count) break;
    uint64_t* o = a.acc + ((size_t)(i0 + c) * 2 * a.nt + t) * N + eo;
#pragma unroll
    for (int p = 0; p < 2; ++p) {
      uint64_t r2[2];
#pragma unroll
      for (int u = 0; u < 2; ++u) {
        if (split) {
          r2[u] = split3_final(ll[c][p][u], hh[c][p][u], ss[c][p][u], sb, pr, p == 0 && add_c0, s0[c][u], pm);
        } else {
          uint64_t lo = ll[c][p][u], hi = hh[c][p][u];
          if (p == 0 && add_c0) mac128(lo, hi, reduce64(s0[c][u], pr), pm);
          r2[u] = reduce128_any(hi, lo, pr);
        }
      }
      *reinterpret_cast<ulonglong2*>(o + (size_t)p * a.nt * N) = make_ulonglong2(r2[0], r2[1]);
    }
  }
}

// ---- ModDown, fused the same way ------------------------------------------
// The P-part of the accumulators (coefficient form after its inverse NTT,
// whose column pass md_conv_col runs itself when only the row pass was run
// before it) is converted to each target limb inside the load of the forward
// NTT's column pass (as k_moddown_conv: conv = BConv(y + h) - h), and the row pass ends
// with the combine of k_ks_combine: out = add + (acc_Q - NTT(conv)) * P^-1.
// A CTA handles both parts of one ciphertext for one limb and tile, so the
// staged twiddles serve two transforms.
struct MdArgs {
  // The P part (coefficient form): ciphertext i, part p, special prime u at
  // yP + i*yp_stride + p*yp_pstride + u*N.
  const uint64_t* yP;
  uint64_t yp_stride, yp_pstride;
  CtBatch accq;         // the Q part (evaluation form), limbs 0 .. level-1
  uint64_t* conv;       // count x [2][level][N]: column-pass outputs
  CtBatch add, out;
  int has_add;          // 0 none, 1 part 0 only, 2 both parts, 3 permuted on part 0 plus plain on both
  uint32_t n_gal;       // part 0 of the addend is added through each automorphism X -> X^gal[g]
  uint64_t gal[HE_MAX_ROT];
  uint32_t level, alpha, L;
  uint32_t spr[HE_MAX_DIGIT];  // prime indices of the alpha dropped limbs (the special primes; q_l for a
                               // rescale by q_l; q_{l-1} and the special primes for a ModDown merged with it)
  // a rescale of k times the input (kind 1 with scaled set): k modulo the target
  // limbs (Shoup pairs) and, times N^-1 where the inverse transform is finished
  // here, modulo the dropped one; k0 (with_k0) is added to part 0
  int scaled, with_k0;
  uint64_t src_w, src_wsh;
  uint64_t kw[HE_MAX_PRIMES], kwsh[HE_MAX_PRIMES], k0[HE_MAX_PRIMES];
  int kind;                    // 0 ModDown, 1 rescale, 2 ModDown merged with the rescale (profile names)
  const uint64_t* addw;        // the addend is multiplied by these Shoup pairs per target limb (nullptr: not)
  const PrimeDev* primes;
  const ulonglong2* tw;
  const ulonglong2* itw;  // inverse twiddles (half)
  int half;               // yP holds only the inverse transform's row pass: md_conv_col finishes it
  uint32_t splits;        // CTAs of md_conv_col that share one tile's target limbs
  int part_ctas;          // md_row_combine: a CTA per part instead of both parts in turn
  const uint64_t* md;   // ModDown tables (params.cu)
};

// Grid: count * 2 * splits * TILES; the conversion's per-special-prime terms
// and the multiple v of P are computed once per element and kept in shared
// memory ([alpha][TILE] words and [TILE] counts) for the CTA's share of the
// level target limbs, which its G groups of T threads take in turn (as in
// ks_modup_col_all).
template <int LOG_N, int LOG_M, int LOG_K, int G, bool SPLIT>
__global__ void __launch_bounds__(G * ((1 << (LOG_M + LOG_K)) / 8), 1024 / (G * ((1 << (LOG_M + LOG_K)) / 8)))
md_conv_col(MdArgs a) {
  using S = Shape<LOG_N, LOG_M, LOG_K, true>;
  constexpr uint32_t N = 1u << LOG_N, TW = S::TILE + S::TILE / 8;
  extern __shared__ __align__(16) unsigned char smem_raw[];
  const uint32_t grp = G == 1 ? 0u : threadIdx.x / S::T, tid = G == 1 ? threadIdx.x : threadIdx.x % S::T;
  ulonglong2* stw = reinterpret_cast<ulonglong2*>(smem_raw) + grp * S::NTW;
  uint64_t* sm0 = reinterpret_cast<uint64_t*>(smem_raw + sizeof(ulonglong2) * S::NTW * G);
  uint64_t* sm = sm0 + grp * TW;
  uint64_t* wv = sm0 + G * TW;                                                  // [alpha][TILE]
  uint32_t* vv = reinterpret_cast<uint32_t*>(wv + (size_t)a.alpha * S::TILE);  // [TILE]
  uint32_t b = blockIdx.x;
  const uint32_t tile = b % S::TILES;
  b /= S::TILES;
  const uint32_t part = b % a.splits;
  b /= a.splits;
  const uint32_t p = b % 2, i = b / 2;
  const uint32_t t_end = (part + 1) * a.level / a.splits;
  const uint64_t* mat = a.md + 2 * a.alpha;
  const uint64_t* hP = mat + (size_t)a.alpha * a.L + 2 * a.L;
  const uint64_t* mat_sh = hP + a.alpha + a.L;
  const uint64_t* wlo = mat_sh + (size_t)a.alpha * a.L;
  const uint64_t* phat = wlo + a.alpha + 9 * (size_t)a.L;         // [alpha][8] words of P/p_u, then [8] of P
  const uint64_t* mat_2 = phat + 8 * (size_t)a.alpha + 8;         // (alpha > 1)
  const uint64_t* yP = a.yP + (size_t)i * a.yp_stride + (size_t)p * a.yp_pstride;
  const bool halves = SPLIT && a.alpha > 1;
  // exact conversion: sum_u w_u (P/p_u) - v P, w_u = [y_u (P/p_u)^-1]_{p_u},
  // v = floor(sum_u w_u / p_u) (64.64 fixed point, resolved exactly near an
  // integer)
  for (uint32_t u = grp; u < a.alpha; u += G) {
    const PrimeDev pp = a.primes[a.spr[u]];
    const uint64_t* src = yP + (size_t)u * N;
    if (a.half) {
      // the inverse transform's column pass on this tile, then the scaling by N^-1
      stage_twiddles<LOG_N, LOG_M, LOG_K, true>(stw, a.itw + (size_t)a.spr[u] * N, tile, tid, S::T);
      pdl_wait();
#pragma unroll 8
      for (uint32_t idx = tid; idx < (uint32_t)S::TILE; idx += S::T)
        sm[idx + (idx >> 3)] = src[S::gidx(tile, idx & (S::K - 1), idx >> LOG_K)];
      group_sync<G, S::T>(grp);
      run_rounds<true, LOG_N, LOG_M, LOG_K, true, 3, G>(sm, stw, pp, tid, grp);
    }
    pdl_wait();
    // the thread's words of the limb first (eight loads in flight), then their products
    uint64_t y0[S::TILE / S::T];
#pragma unroll
    for (int v = 0; v < S::TILE / S::T; ++v) {
      const uint32_t idx = tid + v * S::T;
      y0[v] = a.half ? sm[idx + (idx >> 3)] : src[S::gidx(tile, idx & (S::K - 1), idx >> LOG_K)];
    }
    const uint64_t h = hP[u], w = a.md[2 * u], wsh = a.md[2 * u + 1];
#pragma unroll
    for (int v = 0; v < S::TILE / S::T; ++v) {
      if (a.scaled) y0[v] = mul_shoup(y0[v], a.src_w, a.src_wsh, pp.q);
      else if (a.half) y0[v] = mul_shoup(y0[v], pp.n_inv, pp.n_inv_sh, pp.q);
      const uint64_t x = mul_shoup(add_mod(y0[v], h, pp.q), w, wsh, pp.q);
      wv[(size_t)u * S::TILE + tid + v * S::T] = halves ? split_source(x) : x;
    }
    // the next limb's staging overwrites stw and sm: wait for every thread
    if (a.half) group_sync<G, S::T>(grp);
  }
  pdl_wait();  // (groups without a source)
  if (G > 1) __syncthreads();  // every group's sources
#pragma unroll 2
  for (uint32_t idx = threadIdx.x; idx < (uint32_t)S::TILE; idx += G * S::T) {
    uint64_t fs = 0;
    uint32_t v = 0;
    if (a.alpha > 1) {
      for (uint32_t u = 0; u < a.alpha; ++u) {
        const uint64_t x = wv[(size_t)u * S::TILE + idx];
        frac_acc(halves ? join_source(x) : x, a.primes[a.spr[u]].one_sh, wlo[u], &fs, &v);
      }
      if (frac_in_window(fs, a.alpha))
        v = exact_lift_multiple(wv + idx, S::TILE, a.alpha, phat, phat + 8 * (size_t)a.alpha, v, halves);
    }
    vv[idx] = v;
  }
  if (G > 1) __syncthreads();
  for (uint32_t t = part * a.level / a.splits + grp; t < t_end; t += G) {
    const PrimeDev pr = a.primes[t];
    const uint64_t hQ = hP[a.alpha + t];
    const uint64_t* vP = wlo + a.alpha + a.L + (size_t)t * 8;  // v P mod q_t, v < 8
    stage_twiddles<LOG_N, LOG_M, LOG_K, true>(stw, a.tw + (size_t)t * N, tile, tid, S::T);
    if (SPLIT)
      conv_split<S::TILE, S::T>(a.alpha, sm, wv, mat + t, mat_2 + t, a.L, pr, tid, vv, vP, hQ);
    else
      conv_sum<S::TILE, S::T>(a.alpha, sm, wv, mat + t, mat_sh + t, a.L, pr, tid, vv, vP, hQ);
    group_sync<G, S::T>(grp);
    run_rounds<false, LOG_N, LOG_M, LOG_K, true, 3, G>(sm, stw, pr, tid, grp);
    uint64_t* out = a.conv + (((size_t)i * 2 + p) * a.level + t) * N;
#pragma unroll 8
    for (uint32_t idx = tid; idx < (uint32_t)S::TILE; idx += S::T) {
      const uint32_t xx = idx >> LOG_K, k = idx & (S::K - 1);
      out[S::gidx(tile, k, xx)] = sm[idx + (idx >> 3)];
    }
  }
}

template <int LOG_N, int LOG_M, int LOG_K>
__global__ void __launch_bounds__((1 << (LOG_M + LOG_K)) / 8, 3) md_row_combine(MdArgs a) {
  using S = Shape<LOG_N, LOG_M, LOG_K, false>;
  constexpr uint32_t N = 1u << LOG_N;
  extern __shared__ __align__(16) unsigned char smem_raw[];
  ulonglong2* stw = reinterpret_cast<ulonglong2*>(smem_raw);
  uint64_t* sm = reinterpret_cast<uint64_t*>(smem_raw + sizeof(ulonglong2) * S::NTW);
  uint32_t b = blockIdx.x;
  const uint32_t tile = b % S::TILES;
  b /= S::TILES;
  const uint32_t t = b % a.level;
  b /= a.level;
  const uint32_t i = a.part_ctas ? b >> 1 : b;
  const PrimeDev pr = a.primes[t];
  const uint64_t q = pr.q;
  const uint64_t* pinv = a.md + 2 * a.alpha + (size_t)a.alpha * a.L;
  const uint64_t w = pinv[2 * t], wsh = pinv[2 * t + 1];
  const uint64_t dw = a.addw ? a.addw[2 * t] : 1, dwsh = a.addw ? a.addw[2 * t + 1] : 0;
  stage_twiddles<LOG_N, LOG_M, LOG_K, false>(stw, a.tw + (size_t)t * N, tile);
  pdl_wait();
  constexpr int PER = S::TILE / S::T;
  for (uint32_t p = 0; p < 2; ++p) {
    if (a.part_ctas && p != (b & 1)) continue;  // (the other part has its own CTA)
    const uint64_t* src = a.conv + (((size_t)i * 2 + p) * a.level + t) * N;
#pragma unroll 8
    for (uint32_t idx = threadIdx.x; idx < (uint32_t)S::TILE; idx += S::T) {
      const uint32_t k = idx >> LOG_M, x = idx & (S::M - 1);
      sm[idx + (idx >> 3)] = src[S::gidx(tile, k, x)];
    }
    // the epilogue's operands are loaded before the transform so that their
    // latency overlaps its rounds
    const uint64_t* accq = cpoly(a.accq, i, p, t, N);
    const bool add = a.has_add >= 2 || (a.has_add == 1 && p == 0);
    const bool add_perm = (a.has_add == 1 || a.has_add == 3) && p == 0 && a.n_gal;  // part 0 through the automorphisms
    const bool add_plain = a.has_add == 3 || (add && !add_perm);                     // the addend as it is
    const uint64_t* ad = add ? cpoly(a.add, i, p, t, N) : nullptr;
    uint64_t av[PER], dv[PER];
#pragma unroll
    for (int u = 0; u < PER; ++u) {
      const uint32_t idx = threadIdx.x + u * S::T;
      const uint32_t e = S::gidx(tile, idx >> LOG_M, idx & (S::M - 1));
      av[u] = accq[e];
      dv[u] = add_plain ? ad[e] : 0;
    }
    if (add_perm)  // one automorphism at a time: the thread's PER gathers are independent loads
      for (uint32_t g = 0; g < a.n_gal; ++g) {
        uint64_t gv[PER];
#pragma unroll
        for (int u = 0; u < PER; ++u) {
          const uint32_t idx = threadIdx.x + u * S::T;
          const uint32_t e = S::gidx(tile, idx >> LOG_M, idx & (S::M - 1));
          gv[u] = ad[automorph_src(e, a.gal[g], LOG_N)];
        }
#pragma unroll
        for (int u = 0; u < PER; ++u) dv[u] = add_mod(dv[u], gv[u], q);
      }
    __syncthreads();
    run_rounds<false, LOG_N, LOG_M, LOG_K, false>(sm, stw, pr, threadIdx.x);
    uint64_t* o = cpoly(a.out, i, p, t, N);
#pragma unroll
    for (int u = 0; u < PER; ++u) {
      const uint32_t idx = threadIdx.x + u * S::T;
      const uint32_t e = S::gidx(tile, idx >> LOG_M, idx & (S::M - 1));
      const uint64_t v = sm[idx + (idx >> 3)];
      const uint64_t cv = fwd_final(v, pr);
      const uint64_t x = a.scaled ? mul_shoup(av[u], a.kw[t], a.kwsh[t], q) : av[u];
      uint64_t r = mul_shoup(sub_mod(x, cv, q), w, wsh, q);
      if (add) r = add_mod(r, a.addw ? mul_shoup(dv[u], dw, dwsh, q) : dv[u], q);
      if (a.with_k0 && p == 0) r = add_mod(r, a.k0[t], q);
      o[e] = r;
    }
  }
}

// Dynamic shared memory of the conversion kernels with ns source limbs (md:
// and the lift's counts) and g groups.
template <int LOG_N, int M1, int K1>
size_t conv_smem(uint32_t ns, bool md, int g) {
  using SC = Shape<LOG_N, M1, K1, true>;
  return (sizeof(ulonglong2) * SC::NTW + sizeof(uint64_t) * (SC::TILE + SC::TILE / 8)) * g +
         (sizeof(uint64_t) * ns + (md ? sizeof(uint32_t) : 0)) * SC::TILE;
}

// How a conversion kernel's target limbs are shared: `blocks` CTAs (digits or
// parts times tiles), each split in `splits`, of `groups` groups of threads.  A
// CTA pays a setup of `setup` units per source limb and then one unit per
// target (a target's conversion and column pass), its groups side by side.  A
// group's chain is bound by latency (a unit takes 4.4 us alone on its SM, 5.9
// beside two others, N = 2^13), so a batch that leaves CTA slots free is split
// as far as they reach; together an SM's groups finish a unit every 2.1 us, so
// the repeated setup must not cost more than the shorter chains give: the time
// is the larger of the chain and 0.48 of the SM's units.  One rotation at N = 2^13, level 19: 20 and
// 8 CTAs walked 19 to 23 targets each, 101 and 122 us, split 25 and 23.
// 288 CTAs of 9 units at N = 2^12 stay as they are: 36 us, split in two 48.
// Groups instead of splits or where the sources leave an SM few CTAs: five
// ciphertexts' step at N = 2^13 1072 us with one group, 999 with two; ModUp of
// eight ciphertexts at N = 2^16 740 and 667.
struct ConvPlan {
  uint32_t splits = 1;
  int groups = 1;
  double cost = 0.0;
  size_t smem = 0;  // 0: no number of groups fits
};
constexpr double kSetupHalf = 1.0, kSetupFull = 0.3;  // (with the inverse column pass; a load and a product)

template <int LOG_N, int M1, int K1>
ConvPlan conv_plan(const he_ctx* c, size_t blocks, uint32_t ns, bool md, uint32_t targets, bool half) {
  using SC = Shape<LOG_N, M1, K1, true>;
  const double per = half ? kSetupHalf : kSetupFull;
  ConvPlan best;
  size_t best_warps = 0;
  for (int g : {1, 2, 4}) {
    const size_t sm = conv_smem<LOG_N, M1, K1>(ns, md, g);
    if (g * SC::T > 1024 || sm > kConvSmemMax || (uint32_t)g > targets) continue;
    const size_t ctas = std::max<size_t>(1, std::min<size_t>(c->smem_per_sm / (sm + 1024), 1024 / (g * SC::T)));
    const size_t warps = ctas * g * SC::T / 32, slots = 152 * ctas;
    for (uint32_t s = 1; s <= targets && (s == 1 || blocks * s <= slots); ++s) {
      const uint32_t chain_t = ((targets + s - 1) / s + g - 1) / g;
      // (groups beside each other slow a chain by 0.35 each: rotation at N = 2^13 97 us with 0.17, 93 with 0.35)
      const double beside = 0.35 * (double)(std::min(ctas, (blocks * s + 151) / 152) * g - 1);
      const size_t waves = (blocks * s + slots - 1) / slots;
      const double chain = (double)waves * (per * ((ns + g - 1) / g) + chain_t) * (waves <= 2 ? 1.0 + beside : 1.0);
      const double cost = std::max(chain, 0.48 / 152 * (double)blocks * (s * per * ns + targets));
      // equal times: more resident warps, then fewer CTAs and groups
      if (!best.smem || cost < best.cost || (cost == best.cost && warps > best_warps)) {
        best = ConvPlan{s, g, cost, sm};
        best_warps = warps;
      }
    }
  }
  return best;
}

// Units a column pass launched by itself costs.
inline double col_pass_units(size_t polys, int tiles) {
  return 1.5 + std::max(1.0, 0.48 / 152 * (double)(polys * tiles));
}

// Whether md_conv_col finishes the dropped limbs' inverse transform itself.
template <int LOG_N, int M1, int K1>
bool md_half(const he_ctx* c, uint32_t nd, uint32_t targets, uint32_t count) {
  using SC = Shape<LOG_N, M1, K1, true>;
  const size_t blocks = (size_t)count * 2 * SC::TILES;
  const ConvPlan half = conv_plan<LOG_N, M1, K1>(c, blocks, nd, true, targets, true);
  const ConvPlan full = conv_plan<LOG_N, M1, K1>(c, blocks, nd, true, targets, false);
  return half.smem && half.cost <= full.cost + col_pass_units((size_t)count * 2 * nd, SC::TILES);
}

template <int LOG_N, int M1, int K1, int M2, int K2>
int md_fused_run(he_ctx* c, const MdArgs& a0, uint32_t count, bool* handled) {
  using SC = Shape<LOG_N, M1, K1, true>;
  MdArgs a = a0;
  uint32_t src_bits = 0;
  for (uint32_t u = 0; u < a.alpha; ++u)
    src_bits = std::max(src_bits, (uint32_t)(64 - __builtin_clzll(c->q[a.spr[u]])));
  bool split = true;  // every target's conversion runs as conv_split_tile
  for (uint32_t t = 0; t < a.level; ++t) split = split && conv_split_ok(c->q[t], a.alpha, src_bits);
  using SR = Shape<LOG_N, M2, K2, false>;
  const ConvPlan plan =
      conv_plan<LOG_N, M1, K1>(c, (size_t)count * 2 * SC::TILES, a.alpha, true, a.level, a.half != 0);
  const size_t smr = sizeof(ulonglong2) * SR::NTW + sizeof(uint64_t) * (SR::TILE + SR::TILE / 8);
  if (!plan.smem) {  // too many special primes for this tile: the caller runs the unfused sequence
    *handled = false;
    if (a.half) return fail(HE_EINVAL, "md_fused: half-transformed input needs the fused kernels");
    return HE_OK;
  }
  *handled = true;
  static std::atomic<unsigned long long> attr_row{0};
  const auto conv_kernel = [&]() -> void (*)(MdArgs) {
    if constexpr (4 * SC::T <= 1024)
      if (plan.groups == 4) return split ? md_conv_col<LOG_N, M1, K1, 4, true> : md_conv_col<LOG_N, M1, K1, 4, false>;
    if (plan.groups == 2) return split ? md_conv_col<LOG_N, M1, K1, 2, true> : md_conv_col<LOG_N, M1, K1, 2, false>;
    return split ? md_conv_col<LOG_N, M1, K1, 1, true> : md_conv_col<LOG_N, M1, K1, 1, false>;
  }();
  static std::atomic<unsigned long long> attr_g[2][3]{};
  HE_TRY(set_smem_attr_once(attr_g[split][plan.groups >> 1], c->device, (const void*)conv_kernel, kConvSmemMax));
  HE_TRY(set_smem_attr_once(attr_row, c->device, (const void*)md_row_combine<LOG_N, M2, K2>, smr));
  const double n = (double)(1u << LOG_N);
  const double polys = 2.0 * count * a.level;  // transformed limbs
  double spolys = 0.0, sdrop = 0.0;            // those, and the dropped ones, with split butterflies
  for (uint32_t t = 0; t < a.level && c->prof_on; ++t) spolys += split_limb(c, t) ? 2.0 * count : 0.0;
  for (uint32_t u = 0; u < a.alpha && c->prof_on; ++u) sdrop += split_limb(c, a.spr[u]) ? 2.0 * count : 0.0;
  const char* nm_col = a.kind == 1 ? "rescale_ntt" : a.kind == 2 ? "moddown_rescale_ntt" : "moddown_ntt";
  const char* nm_row = a.kind == 1 ? "rescale_ntt_final" : a.kind == 2 ? "moddown_rescale_ntt_combine"
                                                                       : "moddown_ntt_combine";
  {
    a.splits = plan.splits;
    const size_t blocks = (size_t)count * 2 * SC::TILES * a.splits;
    // with a half-transformed input, also the dropped limbs' inverse column pass
    const double bfly = polys * n / 2 * M1 + (a.half ? 2.0 * count * a.alpha * n / 2 * M1 : 0.0);
    ProfScope prof(c, nm_col, bfly + polys * n * a.alpha, n * 8 * (2.0 * count * a.alpha + polys), 0.0, bfly, 0.0,
                   (spolys + (a.half ? sdrop : 0.0)) * n / 2 * M1, split ? polys * n * a.alpha : 0.0);
    HE_TRY(launch_pdl(conv_kernel, blocks, plan.groups * SC::T, plan.smem, c->stream,
                      a));
  }
  {
    // both parts in one CTA share its twiddles; in a grid that leaves the chip
    // idle each has its own CTA, half the chain
    a.part_ctas = (size_t)count * a.level * SR::TILES <= 304;
    const size_t blocks = (size_t)count * a.level * SR::TILES * (a.part_ctas ? 2 : 1);
    const double addw = a.has_add == 3 ? 1.5 * polys : a.has_add == 2 ? polys : a.has_add == 1 ? polys / 2 : 0.0;
    ProfScope prof(c, nm_row, polys * (n / 2 * M2 + 2 * n), n * 8 * (3.0 * polys + addw), 0.0, polys * n / 2 * M2,
                   0.0, spolys * n / 2 * M2);
    HE_TRY(launch_pdl((md_row_combine<LOG_N, M2, K2>), blocks, SR::T, smr, c->stream,
                      a));
  }
  return HE_OK;
}

// Whether ks_modup_col_all finishes the input's inverse transform itself.
template <int LOG_N, int M1, int K1>
bool ks_half(const he_ctx* c, uint32_t level, uint32_t beta, uint32_t cnt, uint32_t count) {
  using SC = Shape<LOG_N, M1, K1, true>;
  const size_t blocks = (size_t)count * beta * SC::TILES;
  const uint32_t nt = level + (uint32_t)c->alpha;
  const ConvPlan half = conv_plan<LOG_N, M1, K1>(c, blocks, cnt, false, nt, true);
  const ConvPlan full = conv_plan<LOG_N, M1, K1>(c, blocks, cnt, false, nt, false);
  return half.smem && half.cost <= full.cost + col_pass_units((size_t)count * level, SC::TILES);
}

// Limbs per ciphertext with split butterflies: the converted ones (split) and
// the input's own (all); nothing is counted while the timing is off.
inline LimbCount ks_split_limbs(const he_ctx* c, const KsFusedArgs& a) {
  LimbCount n;
  for (uint32_t t = 0; t < a.nt && c->prof_on; ++t)
    if (split_limb(c, ks_prime(t, a.level, a.L))) {
      n.split += t < a.level ? a.beta - 1 : a.beta;
      n.all += t < a.level ? 1 : 0;
    }
  return n;
}

// The ModUp + column-pass launch shared by the key switch and the hoisted
// rotate-and-sum.
template <int LOG_N, int M1, int K1>
int ks_modup_launch(he_ctx* c, const KsFusedArgs& a0, uint32_t count) {
  KsFusedArgs a = a0;
  uint32_t src_bits = 0;
  for (uint32_t t = 0; t < a.level; ++t) src_bits = std::max(src_bits, (uint32_t)(64 - __builtin_clzll(c->q[t])));
  bool split = true;  // every target's conversion runs as conv_split_tile
  for (uint32_t t = 0; t < a.nt; ++t)
    for (uint32_t j : {0u, a.beta - 1})  // (only the last digit may be shorter)
      split = split && conv_split_ok(c->q[ks_prime(t, a.level, a.L)], a.cnt[j], src_bits);
  using SC = Shape<LOG_N, M1, K1, true>;
  const size_t smc = sizeof(ulonglong2) * SC::NTW + sizeof(uint64_t) * (SC::TILE + SC::TILE / 8);
  static std::atomic<unsigned long long> attr_one{0}, attr_g[2][3]{};
  HE_TRY(set_smem_attr_once(attr_one, c->device, (const void*)ks_modup_col<LOG_N, M1, K1>, smc));
  const double n = (double)(1u << LOG_N);
  double own = 0;  // limbs each ciphertext takes as they are
  for (uint32_t j = 0; j < a.beta; ++j) own += a.cnt[j];
  const double conv = (double)a.beta * a.nt - own;  // converted limbs per ciphertext
  const LimbCount sl = ks_split_limbs(c, a);
  double conv_products = 0;  // basis-conversion products (none when a digit is one limb)
  for (uint32_t j = 0; j < a.beta; ++j)
    if (a.cnt[j] > 1) conv_products += (double)(a.nt - a.cnt[j]) * a.cnt[j];
  // work = modular products: butterflies, conversion products
  {
    // with a half-transformed input the kernel also runs the inverse column pass of the level input limbs
    const double inv_bfly = a.half ? (double)a.level * n / 2 * M1 + (double)a.level * n : 0.0;
    const double bfly = count * (conv * n / 2 * M1 + (a.half ? (double)a.level * n / 2 * M1 : 0.0));
    // (the first digit has the most limbs)
    const ConvPlan plan =
        conv_plan<LOG_N, M1, K1>(c, (size_t)count * a.beta * SC::TILES, a.cnt[0], false, a.nt, a.half != 0);
    ProfScope prof(c, "ks_modup_ntt", count * (conv * n / 2 * M1 + conv_products * n + inv_bfly),
                   count * n * 8 * (a.level + conv), 0.0, bfly, 0.0,
                   count * n / 2 * M1 * (sl.split + (a.half ? sl.all : 0.0)),
                   split && plan.smem ? count * conv_products * n : 0.0);
    if (a.half && !plan.smem) return fail(HE_EINVAL, "ks_fused: half-transformed input needs the all-targets kernel");
    if (plan.smem) {  // the targets of one digit and tile in `splits` CTAs
      const auto kernel = [&]() -> void (*)(KsFusedArgs) {
        if constexpr (4 * SC::T <= 1024)
          if (plan.groups == 4)
            return split ? ks_modup_col_all<LOG_N, M1, K1, 4, true> : ks_modup_col_all<LOG_N, M1, K1, 4, false>;
        if (plan.groups == 2)
          return split ? ks_modup_col_all<LOG_N, M1, K1, 2, true> : ks_modup_col_all<LOG_N, M1, K1, 2, false>;
        return split ? ks_modup_col_all<LOG_N, M1, K1, 1, true> : ks_modup_col_all<LOG_N, M1, K1, 1, false>;
      }();
      HE_TRY(set_smem_attr_once(attr_g[split][plan.groups >> 1], c->device, (const void*)kernel, kConvSmemMax));
      a.splits = plan.splits;
      const size_t blocks = (size_t)count * a.beta * SC::TILES * a.splits;
      HE_TRY(launch_pdl(kernel, blocks, plan.groups * SC::T, plan.smem, c->stream,
                        a));
    } else {
      const size_t blocks = (size_t)count * a.beta * a.nt * SC::TILES;
      HE_TRY(launch_pdl((ks_modup_col<LOG_N, M1, K1>), blocks, SC::T, smc, c->stream,
                        a));
    }
  }
  HE_CUDA(cudaGetLastError());
  return HE_OK;
}

// Dynamic shared memory of ks_row_rot (row tiles of half the row pass's
// tile: M2 x 2^(K2-1)) for beta digits of ct ciphertexts (and their part 0's
// tiles when c0).
template <int LOG_N, int M2, int K2>
size_t ks_rot_smem(uint32_t beta, uint32_t ct = 1, bool c0 = false) {
  using SR = Shape<LOG_N, M2, K2 - 1, false>;
  return sizeof(ulonglong2) * SR::NTW + sizeof(uint64_t) * (SR::TILE + SR::TILE / 8) * (beta + (c0 ? 1 : 0)) * ct;
}



inline uint32_t brev_host(uint32_t x, int bits) {
  uint32_t r = 0;
  for (int i = 0; i < bits; ++i) r |= ((x >> i) & 1u) << (bits - 1 - i);
  return r;
}

// Whether X -> X^gal maps every row tile of the hoisted row pass (2^LOG_K
// rows of 2^LOG_M evaluation points) onto itself.
template <int LOG_N, int LOG_M, int LOG_K>
bool rot_closed(uint64_t gal) {
  for (uint32_t row = 0; row < (1u << (LOG_N - LOG_M)); ++row) {
    const uint32_t e = 2 * brev_host(row << LOG_M, LOG_N) + 1;
    const uint32_t e2 = (uint32_t)(((uint64_t)e * gal) & ((2ull << LOG_N) - 1));
    const uint32_t srow = brev_host((e2 - 1) >> 1, LOG_N) >> LOG_M;
    if ((srow >> LOG_K) != (row >> LOG_K)) return false;
  }
  return true;
}

int ntt2_forward_rows(he_ctx* c, const PolyBatch& b);

// The hoisted rotate-and-sum's ModUp, column pass, row pass and the inner
// products of every rotation.  *handled = false (nothing launched) when the
// digits' tiles do not fit in shared memory; *c0_added: part 0 of the input
// is in the accumulator; *pd_added: so is P d on the merged ModDown's limb.
template <int LOG_N, int M1, int K1, int M2, int K2>
int ks_rot_run(he_ctx* c, const KsRotArgs& ra, uint32_t count, bool* handled, bool* c0_added, bool* pd_added) {
  using SR = Shape<LOG_N, M2, K2 - 1, false>;
  const KsFusedArgs& a = ra.k;
  const size_t smr = ks_rot_smem<LOG_N, M2, K2>(a.beta);
  *handled = smr <= kRotSmemMax;
  if (!*handled) return HE_OK;
  static std::atomic<unsigned long long> attr1{0}, attr2{0}, attr4{0}, attr_d{0}, attr_g1{0}, attr_g2{0};
  HE_TRY(set_smem_attr_once(attr1, c->device, (const void*)ks_row_rot<LOG_N, M2, K2 - 1, 1, 1>, kRotSmemMax));
  HE_TRY(set_smem_attr_once(attr2, c->device, (const void*)ks_row_rot<LOG_N, M2, K2 - 1, 2, 1>, kRotSmemMax));
  HE_TRY(set_smem_attr_once(attr_d, c->device, (const void*)ks_row_rot<LOG_N, M2, K2 - 1, 1, 4>, kRotSmemMax));
  HE_TRY(set_smem_attr_once(attr4, c->device, (const void*)ks_row_rot<LOG_N, M2, K2 - 1, 4, 1>, kRotSmemMax));
  HE_TRY(set_smem_attr_once(attr_g1, c->device, (const void*)ks_gather_rot<LOG_N, 1>, kRotSmemMax));
  HE_TRY(set_smem_attr_once(attr_g2, c->device, (const void*)ks_gather_rot<LOG_N, 2>, kRotSmemMax));
  bool closed = !ra.reduce_each;
  for (uint32_t r = 0; r < ra.nrot && closed; ++r) closed = rot_closed<LOG_N, M2, K2 - 1>(ra.gal[r]);
  // (a key switch, the only caller with a rotated input, rotates by the identity)
  if (!closed && a.gal) return fail(HE_EINVAL, "ks_rot: a rotated input needs rotations that keep each tile's rows");
  HE_TRY((ks_modup_launch<LOG_N, M1, K1>(c, a, count)));
  const double n = (double)(1u << LOG_N);
  double own = 0;
  for (uint32_t j = 0; j < a.beta; ++j) own += a.cnt[j];
  const double conv = (double)a.beta * a.nt - own;
  KsRotArgs rc = ra;
  rc.count = count;
  if (!closed) {  // the row pass by itself, in place (own limbs are read from the input)
    PolyBatch e;
    e.src = a.ext;
    e.dst = a.ext;
    e.src_stride = e.dst_stride = (uint64_t)a.nt << LOG_N;
    e.npolys = count * a.beta;
    e.nl = a.nt;
    e.limb0 = 0;
    e.level = a.level;
    e.skip_alpha = a.alpha;
    e.skip_beta = a.beta;
    HE_TRY(ntt2_forward_rows(c, e));
  }
  // work: the converted limbs' row-pass butterflies (closed stages), one
  // reduction per accumulator residue, and the key products (split sums on the
  // target limbs whose primes allow them, as the kernels decide; 128-bit
  // multiply-accumulates on the others); bytes: the limbs read once, one
  // accumulator written (the rotations' products are summed into it), each
  // rotation's key read once per launch
  double split_limbs = 0;
  uint32_t split_q = 0, qbits = 0;
  for (uint32_t t = 0; t < a.nt; ++t) {
    const uint32_t k = 64 - __builtin_clzll(c->q[ks_prime(t, a.level, a.L)]);
    if (t < a.level) qbits = std::max(qbits, k);
    if (split3_fits(k, ra.nrot * a.beta)) {
      split_limbs += 1;
      split_q += t < a.level ? 1 : 0;
    }
  }
  // part 0 through the rotations: in closed stages whose limbs q_t all take
  // the split sums, when its tile fits beside the digits'; in the others
  // unless nrot residues could exceed 64 bits
  if (closed ? split_q < a.level || ks_rot_smem<LOG_N, M2, K2>(a.beta, 1, true) > kRotSmemMax
             : qbits + (32 - __builtin_clz(ra.nrot)) > 64)
    rc.c0 = nullptr;
  const bool c0 = rc.c0 != nullptr;
  *c0_added = c0;
  const double per_limb = count * 2.0 * ra.nrot * a.beta * n;
  const double macs = per_limb * (a.nt - split_limbs), mac3 = per_limb * split_limbs;
  // (with part 0: nrot additions and one 128-bit product per residue of its limbs, and those limbs read)
  const double c0_work = c0 ? count * (double)a.level * n : 0.0;
  const double bfly = closed ? count * conv * n / 2 * M2 : 0.0;
  ProfScope prof(c, "ks_ntt_rot_products", bfly + count * 2.0 * a.nt * n + macs + mac3 + c0_work,
                 count * n * 8 * (conv + own + 2.0 * a.nt + (c0 ? a.level : 0)) +
                     8.0 * n * ra.nrot * a.beta * 2.0 * a.nt,
                 macs + c0_work, bfly, mac3, closed ? count * ks_split_limbs(c, a).split * n / 2 * M2 : 0.0);
  *pd_added = false;
  if (!closed) {
    const uint32_t ct = count >= 2 ? 2 : 1;  // two ciphertexts per CTA share its key words
    const size_t blocks = (size_t)a.nt * ((count + ct - 1) / ct) * ((1u << LOG_N) / (2 * kGatherThreads));
    const size_t sm = kGatherRing * (ct + 2) * sizeof(uint64_t) * 2 * kGatherThreads;
    if (ct == 2) HE_TRY(launch_pdl((ks_gather_rot<LOG_N, 2>), blocks, kGatherThreads, sm, c->stream,
                      rc));
    else HE_TRY(launch_pdl((ks_gather_rot<LOG_N, 1>), blocks, kGatherThreads, sm, c->stream,
                      rc));
    return HE_OK;
  }
  // ciphertexts per CTA: the knob, else 2 when that keeps as many warps
  // resident per SM as 1 does (a 15-rotation stage of 512 ciphertexts at N =
  // 2^14, 16 warps either way: 9.3 ms against 10.1 ms for 1 and 10.0 ms for
  // 4; six digits at N = 2^16 would fall from 12 to 8 warps, slower)
  uint32_t ct = 1;
  auto warps = [&](uint32_t k) {  // resident warps per SM with k ciphertexts per CTA
    const size_t sm = ks_rot_smem<LOG_N, M2, K2>(a.beta, k, c0) + 1024;  // + the runtime's reserve per CTA
    const size_t by_smem = c->smem_per_sm / sm, by_regs = 4 / k;
    return std::min(by_smem, by_regs) * k * (size_t)SR::T / 32;
  };
  const uint32_t want = c->ks_ct ? (uint32_t)c->ks_ct : 2u;
  for (uint32_t cand : {4u, 2u})
    if (ct == 1 && cand <= want && cand <= count && ks_rot_smem<LOG_N, M2, K2>(a.beta, cand, c0) <= kRotSmemMax &&
        (c->ks_ct || warps(cand) >= warps(1)))
      ct = cand;
  const size_t blocks = (size_t)a.nt * ((count + ct - 1) / ct) * SR::TILES;
  const size_t sm = ks_rot_smem<LOG_N, M2, K2>(a.beta, ct, c0);
  // four digit groups where the grid leaves most of the chip idle
  if (!c->ks_ct && a.beta > 1 && (size_t)a.nt * count * SR::TILES <= kDigitGroupCtas) {
    *pd_added = true;
    const size_t one_ct = (size_t)a.nt * count * SR::TILES, sm1 = ks_rot_smem<LOG_N, M2, K2>(a.beta, 1, c0);
    return launch_pdl((ks_row_rot<LOG_N, M2, K2 - 1, 1, 4>), one_ct, 4 * SR::T, sm1, c->stream, rc);
  }
  if (ct == 4) HE_TRY(launch_pdl((ks_row_rot<LOG_N, M2, K2 - 1, 4, 1>), blocks, 4 * SR::T, sm, c->stream,
                    rc));
  else if (ct == 2) HE_TRY(launch_pdl((ks_row_rot<LOG_N, M2, K2 - 1, 2, 1>), blocks, 2 * SR::T, sm, c->stream,
                   rc));
  else HE_TRY(launch_pdl((ks_row_rot<LOG_N, M2, K2 - 1, 1, 1>), blocks, SR::T, sm, c->stream,
                    rc));
  return HE_OK;
}

// Per ring size (ks_fused_n12.cu .. ks_fused_n16.cu: one translation unit
// each, so that the template instances compile in parallel): the launches
// for the tile shape c->ntt_shape.
#define HE_KS_FUSED_DECL(NN)                                                         \
  int ks_rot_n##NN(he_ctx* c, const KsRotArgs& a, uint32_t count, bool* handled, bool* c0_added, \
                 bool* pd_added);                                                      \
  size_t ks_rot_smem_n##NN(const he_ctx* c, uint32_t beta);                          \
  int md_fused_n##NN(he_ctx* c, const MdArgs& a, uint32_t count, bool* handled);     \
  bool md_half_n##NN(const he_ctx* c, uint32_t nd, uint32_t targets, uint32_t count); \
  bool ks_half_n##NN(const he_ctx* c, uint32_t level, uint32_t beta, uint32_t cnt, uint32_t count);
HE_KS_FUSED_DECL(12)
HE_KS_FUSED_DECL(13)
HE_KS_FUSED_DECL(14)
HE_KS_FUSED_DECL(15)
HE_KS_FUSED_DECL(16)
#undef HE_KS_FUSED_DECL
#define HE_KS_FUSED_DEFINE(NN)                                                                             \
  int ks_rot_n##NN(he_ctx* c, const KsRotArgs& a, uint32_t count, bool* handled, bool* c0_added,           \
                 bool* pd_added) {                                                                         \
    return with_pair<NN>(c->ntt_shape, [&](auto p) {                                                       \
      return ks_rot_run<NN, p.m1, p.k1, p.m2, p.k2>(c, a, count, handled, c0_added, pd_added);             \
    });                                                                                                    \
  }                                                                                                        \
  size_t ks_rot_smem_n##NN(const he_ctx* c, uint32_t beta) {                                               \
    return with_pair<NN>(c->ntt_shape, [&](auto p) { return ks_rot_smem<NN, p.m2, p.k2>(beta); });         \
  }                                                                                                        \
  int md_fused_n##NN(he_ctx* c, const MdArgs& a, uint32_t count, bool* handled) {                          \
    return with_pair<NN>(c->ntt_shape, [&](auto p) {                                                       \
      return md_fused_run<NN, p.m1, p.k1, p.m2, p.k2>(c, a, count, handled);                               \
    });                                                                                                    \
  }                                                                                                        \
  bool md_half_n##NN(const he_ctx* c, uint32_t nd, uint32_t targets, uint32_t count) {                     \
    return with_pair<NN>(c->ntt_shape, [&](auto p) { return md_half<NN, p.m1, p.k1>(c, nd, targets, count); }); \
  }                                                                                                        \
  bool ks_half_n##NN(const he_ctx* c, uint32_t level, uint32_t beta, uint32_t cnt, uint32_t count) {       \
    return with_pair<NN>(c->ntt_shape, [&](auto p) { return ks_half<NN, p.m1, p.k1>(c, level, beta, cnt, count); }); \
  }

}  // namespace he
