// Expensive-potential kernels in float for n <= 16 (k_ace.cuh).
#include "k_ace.cuh"

namespace mixd {

const AceOps<float> ace_f32_n16 = ace_f32_ops<16>();

}  // namespace mixd
