// Expensive-potential kernels with the bf16 hi/lo tensor-core readout for n <= 12 (k_ace_tc.cuh).
#include "k_ace_tc.cuh"

namespace mixd {

const AceTcOps ace_tc2_n12 = ace_tc_ops<12, 2>();

}  // namespace mixd
