// ntt2_n13.cu -- the compile-time-shaped NTT instantiated for N = 2^13.
#include "ntt2_impl.cuh"

namespace he {

HE_NTT2_DEFINE(13)

}  // namespace he
