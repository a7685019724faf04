// ks_fused_n15.cu -- the fused key-switching kernels instantiated for N = 2^15
// (the three tile shapes of tile_pairs.h).
#include "ks_fused.cuh"

namespace he {

HE_KS_FUSED_DEFINE(15)

}  // namespace he
