// Expensive-potential kernels with the bf16 tensor-core readout for n <= 12 (k_ace_tc.cuh).
#include "k_ace_tc.cuh"

namespace mixd {

const AceTcOps ace_tc1_n12 = ace_tc_ops<12, 1>();

}  // namespace mixd
