// ntt2_n12.cu -- the compile-time-shaped NTT instantiated for N = 2^12.
#include "ntt2_impl.cuh"

namespace he {

HE_NTT2_DEFINE(12)

}  // namespace he
