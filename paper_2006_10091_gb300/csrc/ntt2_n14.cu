// ntt2_n14.cu -- the compile-time-shaped NTT instantiated for N = 2^14.
#include "ntt2_impl.cuh"

namespace he {

HE_NTT2_DEFINE(14)

}  // namespace he
