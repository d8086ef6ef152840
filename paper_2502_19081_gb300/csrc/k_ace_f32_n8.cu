// Expensive-potential kernels in float for n <= 8 (k_ace.cuh).
#include "k_ace.cuh"

namespace mixd {

const AceOps<float> ace_f32_n4 = ace_f32_ops<4>();
const AceOps<float> ace_f32_n8 = ace_f32_ops<8>();

}  // namespace mixd
