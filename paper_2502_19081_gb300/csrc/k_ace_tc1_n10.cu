// Expensive-potential kernels with the bf16 tensor-core readout for n <= 10 (k_ace_tc.cuh).
#include "k_ace_tc.cuh"

namespace mixd {

const AceTcOps ace_tc1_n10 = ace_tc_ops<10, 1>();

}  // namespace mixd
