// ntt2_n15.cu -- the compile-time-shaped NTT instantiated for N = 2^15.
#include "ntt2_impl.cuh"

namespace he {

HE_NTT2_DEFINE(15)

}  // namespace he
