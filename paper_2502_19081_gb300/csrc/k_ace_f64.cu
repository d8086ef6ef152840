// Expensive-potential kernels in float64 (k_ace.cuh), and the dispatch of every
// expensive kernel over precision and class of n (k_ace_ops.h).
#include "k_ace.cuh"

namespace mixd {

namespace {

const AceOps<float>* const OPS_F32[5] = {&ace_f32_n4, &ace_f32_n8, &ace_f32_n10, &ace_f32_n12, &ace_f32_n16};
const AceTcOps* const OPS_TC[2][5] = {{&ace_tc1_n4, &ace_tc1_n8, &ace_tc1_n10, &ace_tc1_n12, &ace_tc1_n16},
                                      {&ace_tc2_n4, &ace_tc2_n8, &ace_tc2_n10, &ace_tc2_n12, &ace_tc2_n16}};

// float64 takes its unit block at run time (QB = 0): n <= 10 shares the class of 12
template <int NP>
constexpr AceOps<double> f64_ops() {
    return {ace_cfg_l<double, NP, 0>, ace_launch_l<double, NP, 0>, ace_batch_launch_l<double, NP, 0>, nullptr};
}
const AceOps<double> OPS_F64[5] = {f64_ops<4>(), f64_ops<8>(), f64_ops<12>(), f64_ops<12>(), f64_ops<16>()};

cudaError_t cfg(int precision, bool batch, int L, int n, int cap, int tile_max, int qb, size_t* smem, int* grid,
                int wn) {
    const int k = ace_class(n);
    return precision == MIX_FP64 ? OPS_F64[k].cfg(batch, L, n, cap, tile_max, qb, smem, grid, wn)
                                 : OPS_F32[k]->cfg(batch, L, n, cap, tile_max, qb, smem, grid, wn);
}

}  // namespace

cudaError_t ace_configure(int precision, int L, int n, int cap, int tile_max, int qb, size_t* smem, int* grid,
                          int wn) {
    if (cap > MAX_CAP || n > 16 || qb < 1 || (wn != ACE_GROUP && wn != ACE_MAX_WARPS)) return cudaErrorInvalidValue;
    return cfg(precision, false, L, n, cap, tile_max, qb, smem, grid, wn);
}

void launch_ace(const Dev& d, const void* tab, int precision, int L, size_t smem, int grid, int wn, cudaStream_t s) {
    if (precision == MIX_FP64) {
        const AceTab<double>& t = *static_cast<const AceTab<double>*>(tab);
        OPS_F64[ace_class(t.n)].launch(d, t, L, smem, grid, wn, s);
    } else {
        const AceTab<float>& t = *static_cast<const AceTab<float>*>(tab);
        OPS_F32[ace_class(t.n)]->launch(d, t, L, smem, grid, wn, s);
    }
}

cudaError_t ace_batch_configure(int precision, int L, int n, int cap, int tile_max, int qb, size_t* smem, int* grid) {
    if (cap > MAX_CAP || n > 16 || qb < 1) return cudaErrorInvalidValue;
    return cfg(precision, true, L, n, cap, tile_max, qb, smem, grid, ACE_GROUP);
}

void launch_ace_batch(int precision, const Dev* devs, const void* tabs, const int2* list, const int* count,
                      int n, int L, size_t smem, int grid, cudaStream_t s) {
    if (precision == MIX_FP64)
        OPS_F64[ace_class(n)].launch_batch(
            AceBatch<double>{devs, static_cast<const AceTab<double>*>(tabs), list, count}, L, smem, grid, s);
    else
        OPS_F32[ace_class(n)]->launch_batch(
            AceBatch<float>{devs, static_cast<const AceTab<float>*>(tabs), list, count}, L, smem, grid, s);
}

cudaError_t ace_tc_configure(int tcm, int L, int n, int cap, int tile_max, int qb, size_t* smem, int* grid,
                             int* nbuf) {
    if (cap > MAX_CAP || n > 16 || qb < 1 || L < 0 || L > 6 || tcm < 1 || tcm > 2) return cudaErrorInvalidValue;
    return OPS_TC[tcm - 1][ace_class(n)]->cfg(L, n, cap, tile_max, qb, smem, grid, nbuf);
}

void launch_ace_tc(const Dev& d, const void* tab, int tcm, int L, size_t smem, int grid, int nbuf, cudaStream_t s) {
    const AceTab<float>& t = *static_cast<const AceTab<float>*>(tab);
    OPS_TC[tcm - 1][ace_class(t.n)]->launch(d, t, L, smem, grid, nbuf, s);
}

cudaError_t ace_gaunt_upload(int tcm, int n_rad, const float* g, int n) {
    const int k = ace_class(n_rad);
    return tcm == 0 ? OPS_F32[k]->upload(g, n) : OPS_TC[tcm - 1][k]->upload(g, n);
}

}  // namespace mixd
