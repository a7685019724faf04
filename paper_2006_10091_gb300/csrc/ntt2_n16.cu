// ntt2_n16.cu -- the compile-time-shaped NTT instantiated for N = 2^16.
#include "ntt2_impl.cuh"

namespace he {

HE_NTT2_DEFINE(16)

}  // namespace he
