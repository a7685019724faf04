// ks_fused_n13.cu -- the fused key-switching kernels instantiated for N = 2^13
// (the three tile shapes of tile_pairs.h).
#include "ks_fused.cuh"

namespace he {

HE_KS_FUSED_DEFINE(13)

}  // namespace he
