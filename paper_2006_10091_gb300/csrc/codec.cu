// codec.cu -- encode/decode (Sec. 3: canonical embedding) and decryption.
//
// Slot j is the value at zeta_j = w^(e_j), w = exp(i pi / N), e_j = 5^j mod
// 2N; its conjugate sits at w^(2N - e_j).  With u(t) = (t - 1)/2 for odd t:
//  encode: coefficient i = (Delta/N) Re(w^-i * F(W)[i]), F the forward
//          (e^-) length-N DFT of W[u(e_j)] = z_j, W[u(2N - e_j)] = conj(z_j),
//          rounded half away from zero;
//  decode: z_j = (1/Delta) G(m w^i)[u(e_j)], G the e^+ length-N DFT.
// Decrypt: m = c0 + c1 s per limb, inverse NTT, Garner's mixed-radix digits,
// centered against (Q-1)/2, converted to double by Horner from the top digit.
#include <math.h>

#include <vector>

#include "he_internal.h"
#include "he_kernels.h"
#include "he_ops.h"

namespace he {

// ---- radix-2 complex FFT in double, two launches -------------------------------
// Decimation in time on the bit-reversed input: stage with half-size h pairs
// (p, p + h) in blocks of 2h with the twiddle exp(sign i pi (p mod h) / h).
// The first launch runs the stages inside contiguous blocks of 2^m1 points
// (m1 = ceil(log2(N)/2)) and reads its input where it lies (the encoder's
// slots through slot_of, the decoder's coefficients with their twist), the
// second runs the rest on kFftCols neighbouring columns and writes the result
// (rounded coefficients, or the slots' values).  A CTA holds few points, one
// butterfly per thread and stage: the double-precision rate of an SM is low, so
// the work is spread wide.  Twiddles come from the context's table (the same
// values, computed once): N = 2^12 forward 69 us in 12 launches of one stage
// each with sincospi per butterfly.
constexpr int kFftCols = 2;

// tab[i] = (cos, sin)(pi i / N); slot_of[u] = j for the point w^(2u+1) of slot j
// (2u + 1 = 5^j mod 2N), -1 - j for its conjugate's.
__global__ void k_codec_tables(double2* tab, int32_t* slot_of, int log_n) {
  const uint32_t n = 1u << log_n, m = 2 * n;
  for (uint32_t i = blockIdx.x * blockDim.x + threadIdx.x; i < n; i += gridDim.x * blockDim.x) {
    double sn, cs;
    sincospi((double)i / (double)n, &sn, &cs);
    tab[i] = make_double2(cs, sn);
    if (i < n / 2) {
      uint32_t e = 1, b = 5, x = i;  // 5^i mod 2N by square-and-multiply
      while (x) {
        if (x & 1) e = (uint32_t)(((uint64_t)e * b) & (m - 1));
        b = (uint32_t)(((uint64_t)b * b) & (m - 1));
        x >>= 1;
      }
      slot_of[(e - 1) / 2] = (int32_t)i;
      slot_of[(m - e - 1) / 2] = -1 - (int32_t)i;
    }
  }
}

int codec_tables(he_ctx* c) {
  const size_t n = c->n;
  HE_CUDA(cudaMalloc(&c->d_fft, sizeof(double2) * n));
  HE_CUDA(cudaMalloc(&c->d_slot_of, sizeof(int32_t) * n));
  k_codec_tables<<<grid_for(n), 256>>>((double2*)c->d_fft, c->d_slot_of, c->log_n);
  HE_CUDA(cudaGetLastError());
  return HE_OK;
}

struct FftArgs {
  const double* in;      // slots (encode: nz of them) or coefficients (decode)
  double2* mid;          // between the passes, N points
  const double2* tab;
  const int32_t* slot_of;
  int64_t* coeffs;       // encode: the result
  int* overflow;         // encode: set when a coefficient leaves int64
  double* re;            // decode: the result (nz slots)
  uint32_t nz;
  double scale;
  int log_n, m1;
};

// sign of the exponent: -1 encode, +1 decode.  The negated sine is kept opaque to
// the compiler: folded into the products it changes which of the two a fused
// multiply-add rounds, and with it last bits and, rarely, a rounded coefficient.
template <bool ENC>
__device__ __forceinline__ double signed_sine(double2 w) {
  double sn = ENC ? -w.y : w.y;
  if (ENC) asm("" : "+d"(sn));
  return sn;
}
template <bool ENC>
__device__ __forceinline__ void fft_butterfly(double2* sm, uint32_t i0, uint32_t i1, double2 w) {
  const double cs = w.x, sn = signed_sine<ENC>(w);
  const double2 x = sm[i0], y = sm[i1];
  const double2 ty = make_double2(y.x * cs - y.y * sn, y.x * sn + y.y * cs);
  sm[i0] = make_double2(x.x + ty.x, x.y + ty.y);
  sm[i1] = make_double2(x.x - ty.x, x.y - ty.y);
}

// Stages h = 1 .. 2^(m1-1) on the block of 2^m1 points blockIdx.x.
template <bool ENC>
__global__ void k_fft_first(FftArgs a) {
  pdl_wait();
  extern __shared__ double2 fsm[];
  const uint32_t m = 1u << a.m1, base = blockIdx.x << a.m1;
  for (uint32_t x = threadIdx.x; x < m; x += blockDim.x) {
    const uint32_t i = brev_bits(base | x, a.log_n);
    if (ENC) {
      const int32_t sl = a.slot_of[i];
      const uint32_t j = (uint32_t)(sl < 0 ? -1 - sl : sl);
      fsm[x] = make_double2(j < a.nz ? a.in[j] : 0.0, 0.0);
    } else {
      const double2 w = a.tab[i];
      const double v = a.in[i];
      fsm[x] = make_double2(v * w.x, v * w.y);
    }
  }
  __syncthreads();
  for (int s = 0; s < a.m1; ++s) {
    const uint32_t h = 1u << s;
    for (uint32_t g = threadIdx.x; g < m / 2; g += blockDim.x) {
      const uint32_t pos = g & (h - 1), i0 = ((g >> s) << (s + 1)) | pos;
      fft_butterfly<ENC>(fsm, i0, i0 + h, a.tab[pos << (a.log_n - s)]);
    }
    __syncthreads();
  }
  for (uint32_t x = threadIdx.x; x < m; x += blockDim.x) a.mid[base | x] = fsm[x];
}

// The remaining stages on columns [kFftCols blockIdx.x, ...): points x 2^m1 + f.
template <bool ENC>
__global__ void k_fft_second(FftArgs a) {
  pdl_wait();
  extern __shared__ double2 fsm[];
  const uint32_t n = 1u << a.log_n;
  const int m2 = a.log_n - a.m1;
  const uint32_t pts = (uint32_t)kFftCols << m2, f0 = blockIdx.x * kFftCols;
  for (uint32_t q = threadIdx.x; q < pts; q += blockDim.x)
    fsm[q] = a.mid[((q / kFftCols) << a.m1) | (f0 + q % kFftCols)];
  __syncthreads();
  for (int s = 0; s < m2; ++s) {
    const uint32_t h = 1u << s;
    for (uint32_t g = threadIdx.x; g < pts / 2; g += blockDim.x) {
      const uint32_t f = g % kFftCols, x = g / kFftCols, pos = x & (h - 1);
      const uint32_t i0 = ((((x >> s) << (s + 1)) | pos) * kFftCols) + f;
      const uint32_t gp = (pos << a.m1) | (f0 + f);  // position within the stage's block of 2^(m1+s+1)
      fft_butterfly<ENC>(fsm, i0, i0 + h * kFftCols, a.tab[gp << (m2 - s)]);
    }
    __syncthreads();
  }
  for (uint32_t q = threadIdx.x; q < pts; q += blockDim.x) {
    const uint32_t i = ((q / kFftCols) << a.m1) | (f0 + q % kFftCols);
    const double2 v = fsm[q];
    if (ENC) {
      const double cs = a.tab[i].x, sn = signed_sine<true>(a.tab[i]);  // w^-i
      const double re = v.x * cs - v.y * sn;
      const double raw = (a.scale / (double)n) * re;
      if (!(fabs(raw) < 9.2e18)) {
        *a.overflow = 1;
        a.coeffs[i] = 0;
      } else {
        a.coeffs[i] = llround(raw);
      }
    } else {
      const int32_t j = a.slot_of[i];
      if (j >= 0 && (uint32_t)j < a.nz) a.re[j] = v.x / a.scale;
    }
  }
}

template <bool ENC>
static int fft_run(he_ctx* c, FftArgs a) {
  a.log_n = c->log_n;
  a.m1 = (c->log_n + 1) / 2;
  a.tab = (const double2*)c->d_fft;
  a.slot_of = c->d_slot_of;
  const uint32_t p1 = 1u << a.m1, p2 = (uint32_t)kFftCols << (c->log_n - a.m1);
  HE_TRY(launch_pdl(k_fft_first<ENC>, c->n / p1, p1 / 2, sizeof(double2) * p1, c->stream,
                    a));
  HE_TRY(launch_pdl(k_fft_second<ENC>, c->n / p2, p2 / 2, sizeof(double2) * p2, c->stream,
                    a));
  return HE_OK;
}

// Encode device slots d_z (n_slots doubles) into device int64 coefficients
// d_out.  scratch: N double2; d_ovf: one int (set when a coefficient leaves int64).
int encode_dev(he_ctx* c, const double* d_z, size_t n_slots, double scale, int64_t* d_out,
               double2* scratch, int* d_ovf) {
  if (n_slots > (size_t)c->n / 2) return fail(HE_EINVAL, "more slots than N/2");
  if (!(scale > 0.0)) return fail(HE_EINVAL, "scale must be positive");
  FftArgs a{};
  a.in = d_z;
  a.mid = scratch;
  a.coeffs = d_out;
  a.overflow = d_ovf;
  a.nz = (uint32_t)n_slots;
  a.scale = scale;
  return fft_run<true>(c, a);
}

// ---- decryption -----------------------------------------------------------------
__global__ void k_decrypt_dot(CtBatch A, const uint64_t* s, uint64_t* m, uint32_t level, int log_n,
                              const PrimeDev* primes) {
  pdl_wait();
  const uint32_t n = 1u << log_n;
  const size_t total = (size_t)level * n;
  for (size_t g = blockIdx.x * (size_t)blockDim.x + threadIdx.x; g < total; g += (size_t)gridDim.x * blockDim.x) {
    const uint32_t t = (uint32_t)(g / n), k = (uint32_t)(g % n);
    const PrimeDev pr = primes[t];
    const uint64_t c0 = A.base[(size_t)t * n + k], c1 = A.base[((size_t)A.cap + t) * n + k];
    m[g] = add_mod(c0, mul_mod(c1, s[(size_t)t * n + k], pr), pr.q);
  }
}

struct GarnerArgs {
  uint64_t half[HE_MAX_PRIMES];  // mixed-radix digits of (Q-1)/2
};

// gar: [L] Shoup pairs of (q_0..q_{i-1})^-1 mod q_i, then [L][L] prefix products
// (q_0..q_{i'-1}) mod q_i at [i][i'].
__global__ void k_crt_double(const uint64_t* m, double* out, uint32_t level, int log_n,
                             const PrimeDev* primes, const uint64_t* gar, uint32_t L, GarnerArgs ga) {
  pdl_wait();
  const uint32_t n = 1u << log_n;
  for (uint32_t k = blockIdx.x * blockDim.x + threadIdx.x; k < n; k += gridDim.x * blockDim.x) {
    uint64_t d[HE_MAX_PRIMES];
    for (uint32_t i = 0; i < level; ++i) {
      const PrimeDev pr = primes[i];
      const uint64_t* pref = gar + 2 * L + (size_t)i * L;
      uint64_t acc = 0;
      for (uint32_t j = 0; j < i; ++j) acc = add_mod(acc, mul_mod(reduce64(d[j], pr), pref[j], pr), pr.q);
      const uint64_t x = sub_mod(m[(size_t)i * n + k], acc, pr.q);
      d[i] = i ? mul_shoup(x, gar[2 * i], gar[2 * i + 1], pr.q) : x;
    }
    int cmp = 0;
    for (int i = (int)level - 1; i >= 0 && cmp == 0; --i)
      cmp = d[i] > ga.half[i] ? 1 : (d[i] < ga.half[i] ? -1 : 0);
    const bool neg = cmp > 0;
    if (neg) {  // Q - v = (Q - 1 - v) + 1
      uint64_t carry = 1;
      for (uint32_t i = 0; i < level; ++i) {
        uint64_t v = primes[i].q - 1 - d[i] + carry;
        carry = 0;
        if (v == primes[i].q) { v = 0; carry = 1; }
        d[i] = v;
      }
    }
    double v = (double)d[level - 1];
    for (int i = (int)level - 2; i >= 0; --i) v = v * (double)primes[i].q + (double)d[i];
    out[k] = neg ? -v : v;
  }
}

// scratch m: level*N words.
int decrypt_dev(he_ctx* c, const he_ct* ct, uint64_t* m, double* d_coeffs) {
  const uint32_t n = c->n, level = ct->level;
  const size_t lw = (size_t)level * n;
  CtBatch A{ct->data, 0, ct->cap, 0};
  HE_TRY(launch_pdl(k_decrypt_dot, grid_for(lw), 256, 0, c->stream,
                    A, c->d_s, m, level, c->log_n, c->d_primes));
  PolyBatch b;
  b.src = m;
  b.dst = m;
  b.src_stride = b.dst_stride = 0;
  b.npolys = 1;
  b.nl = level;
  b.limb0 = 0;
  b.level = c->L;
  b.skip_alpha = 0;
  b.skip_beta = 1;
  HE_TRY(ntt_inverse(c, b));
  // digits of (Q-1)/2: Q-1 has digits q_i - 1; halve from the top digit down
  GarnerArgs ga;
  unsigned __int128 carry = 0;
  for (int i = (int)level - 1; i >= 0; --i) {
    const unsigned __int128 cur = carry * c->q[i] + (c->q[i] - 1);
    ga.half[i] = (uint64_t)(cur / 2);
    carry = cur % 2;
  }
  HE_TRY(launch_pdl(k_crt_double, grid_for(n), 256, 0, c->stream,
                    m, d_coeffs, level, c->log_n, c->d_primes, c->d_garner, (uint32_t)c->L, ga));
  return HE_OK;
}

// Decode centered coefficients (device doubles d_m) into n_slots device
// values d_re.  scratch: N double2.
int decode_dev(he_ctx* c, const double* d_m, double scale, double* d_re, size_t n_slots,
               double2* scratch) {
  if (n_slots > (size_t)c->n / 2) return fail(HE_EINVAL, "more slots than N/2");
  FftArgs a{};
  a.in = d_m;
  a.mid = scratch;
  a.re = d_re;
  a.nz = (uint32_t)n_slots;
  a.scale = scale;
  return fft_run<false>(c, a);
}

}  // namespace he
