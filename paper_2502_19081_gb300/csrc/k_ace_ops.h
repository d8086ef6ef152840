// The instantiation classes of the expensive kernels.  The float kernels are
// compiled per class of n (the radial functions): N = 4, 8, 10, 12, 16 serve n up
// to N (rows padded to a multiple of 4, the lane units of nu3_qb(N)), a
// translation unit each (4 and 8 share one), because the l-triples of a kernel
// are unrolled and compile slowly; float64 has one unit for all.
#pragma once

#include "mix_launch.h"

namespace mixd {

// Many systems: the flattened list {system, first atom of a group} of one group
// of systems sharing (T, L, class)
template <typename T>
struct AceBatch {
    const Dev* devs;
    const AceTab<T>* tabs;
    const int2* list;
    const int* count;
};

template <typename T>
struct AceOps {
    cudaError_t (*cfg)(bool batch, int L, int n, int cap, int tile_max, int qb, size_t* smem, int* grid, int wn);
    void (*launch)(const Dev& d, const AceTab<T>& tab, int L, size_t smem, int grid, int wn, cudaStream_t s);
    void (*launch_batch)(const AceBatch<T>& b, int L, size_t smem, int grid, cudaStream_t s);
    cudaError_t (*upload)(const float* g, int n);   // Gaunt coefficients into the unit's constant memory (float)
};

struct AceTcOps {
    cudaError_t (*cfg)(int L, int n, int cap, int tile_max, int qb, size_t* smem, int* grid, int* nbuf);
    void (*launch)(const Dev& d, const AceTab<float>& tab, int L, size_t smem, int grid, int nbuf, cudaStream_t s);
    cudaError_t (*upload)(const float* g, int n);
};

// class of n: index into the tables (n <= 4, 8, 10, 12, 16)
inline int ace_class(int n) { return n <= 4 ? 0 : n <= 8 ? 1 : n <= 10 ? 2 : n <= 12 ? 3 : 4; }

extern const AceOps<float> ace_f32_n4, ace_f32_n8, ace_f32_n10, ace_f32_n12, ace_f32_n16;
extern const AceTcOps ace_tc1_n4, ace_tc1_n8, ace_tc1_n10, ace_tc1_n12, ace_tc1_n16;
extern const AceTcOps ace_tc2_n4, ace_tc2_n8, ace_tc2_n10, ace_tc2_n12, ace_tc2_n16;

}  // namespace mixd
