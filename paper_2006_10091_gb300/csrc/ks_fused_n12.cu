// ks_fused_n12.cu -- the fused key-switching kernels instantiated for N = 2^12
// (the three tile shapes of ntt2.cu).
#include "ks_fused.cuh"

namespace he {

int ks_rot_n12(he_ctx* c, const KsRotArgs& a, uint32_t count, bool* handled, bool* c0_added, bool* pd_added) {
  const int sh = c->ntt_shape;
  return sh == 1 ? ks_rot_run<12, 5, 6, 7, 4>(c, a, count, handled, c0_added, pd_added)
       : sh == 2 ? ks_rot_run<12, 3, 8, 9, 2>(c, a, count, handled, c0_added, pd_added) : ks_rot_run<12, 6, 5, 6, 5>(c, a, count, handled, c0_added, pd_added);
}

size_t ks_rot_smem_n12(const he_ctx* c, uint32_t beta) {
  const int sh = c->ntt_shape;
  return sh == 1 ? ks_rot_smem<12, 7, 4>(beta) : sh == 2 ? ks_rot_smem<12, 9, 2>(beta) : ks_rot_smem<12, 6, 5>(beta);
}

int md_fused_n12(he_ctx* c, const MdArgs& a, uint32_t count, bool* handled) {
  const int sh = c->ntt_shape;
  return sh == 1 ? md_fused_run<12, 5, 6, 7, 4>(c, a, count, handled)
       : sh == 2 ? md_fused_run<12, 3, 8, 9, 2>(c, a, count, handled) : md_fused_run<12, 6, 5, 6, 5>(c, a, count, handled);
}

bool md_half_n12(const he_ctx* c, uint32_t nd, uint32_t targets, uint32_t count) {
  const int sh = c->ntt_shape;
  return sh == 1 ? md_half<12, 5, 6>(c, nd, targets, count)
       : sh == 2 ? md_half<12, 3, 8>(c, nd, targets, count) : md_half<12, 6, 5>(c, nd, targets, count);
}

bool ks_half_n12(const he_ctx* c, uint32_t level, uint32_t beta, uint32_t cnt, uint32_t count) {
  const int sh = c->ntt_shape;
  return sh == 1 ? ks_half<12, 5, 6>(c, level, beta, cnt, count)
       : sh == 2 ? ks_half<12, 3, 8>(c, level, beta, cnt, count) : ks_half<12, 6, 5>(c, level, beta, cnt, count);
}

}  // namespace he
