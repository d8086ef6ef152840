// Expensive-potential kernels with the bf16 hi/lo tensor-core readout for n <= 8 (k_ace_tc.cuh).
#include "k_ace_tc.cuh"

namespace mixd {

const AceTcOps ace_tc2_n4 = ace_tc_ops<4, 2>();
const AceTcOps ace_tc2_n8 = ace_tc_ops<8, 2>();

}  // namespace mixd
