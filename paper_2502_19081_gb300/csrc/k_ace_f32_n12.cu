// Expensive-potential kernels in float for n <= 12 (k_ace.cuh).
#include "k_ace.cuh"

namespace mixd {

const AceOps<float> ace_f32_n12 = ace_f32_ops<12>();

}  // namespace mixd
