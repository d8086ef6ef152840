// Expensive-potential kernels in float for n <= 10 (k_ace.cuh).
#include "k_ace.cuh"

namespace mixd {

const AceOps<float> ace_f32_n10 = ace_f32_ops<10>();

}  // namespace mixd
