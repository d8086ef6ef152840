// Expensive-potential kernels with the bf16 hi/lo tensor-core readout for n <= 16 (k_ace_tc.cuh).
#include "k_ace_tc.cuh"

namespace mixd {

const AceTcOps ace_tc2_n16 = ace_tc_ops<16, 2>();

}  // namespace mixd
