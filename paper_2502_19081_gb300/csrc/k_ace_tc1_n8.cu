// Expensive-potential kernels with the bf16 tensor-core readout for n <= 8 (k_ace_tc.cuh).
#include "k_ace_tc.cuh"

namespace mixd {

const AceTcOps ace_tc1_n4 = ace_tc_ops<4, 1>();
const AceTcOps ace_tc1_n8 = ace_tc_ops<8, 1>();

}  // namespace mixd
