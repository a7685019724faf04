// ks_fused_n12.cu -- the fused key-switching kernels instantiated for N = 2^12
// (the three tile shapes of tile_pairs.h).
#include "ks_fused.cuh"

namespace he {

HE_KS_FUSED_DEFINE(12)

}  // namespace he
