// Host-side launchers of the library's kernels (one definition per .cu file).
#pragma once

#include "mix_dev.cuh"

namespace mixd {

// displacement, lists, weights, sets and their compaction in one cooperative
// launch (k_front.cu).  front_configure fills d.grid_front_max.
cudaError_t front_configure(Dev& d);
cudaError_t launch_front(const Dev& d, const Regions& r, const SeedRule& sr, cudaStream_t s, int integrate, double dt,
                         double h, int force_rebuild, bool prof);
// the lists alone, of the positions x_in (copied to d.x and folded there)
cudaError_t launch_front_lists(const Dev& d, const double4* x_in, cudaStream_t s);

// expensive potential (k_ace.cuh, k_ace_f32_n*.cu, k_ace_f64.cu); returns cudaSuccess or the launch error;
// wn: warps (atoms) a CTA, ACE_GROUP or ACE_MAX_WARPS
cudaError_t ace_configure(int precision, int L, int n, int cap, int tile_max, int qb, size_t* smem, int* grid,
                          int wn);
void launch_ace(const Dev& d, const void* tab, int precision, int L, size_t smem, int grid, int wn, cudaStream_t s);

// expensive potential with the tensor-core readout (k_ace_tc.cuh, k_ace_tc*_n*.cu; float tables
// with the bf16 operand sections): tcm 1 bf16, 2 bf16 hi/lo.  *nbuf: tile
// buffers that fit shared memory (2, else 1); cudaErrorInvalidValue when even
// one does not fit
cudaError_t ace_tc_configure(int tcm, int L, int n, int cap, int tile_max, int qb, size_t* smem, int* grid,
                             int* nbuf);
void launch_ace_tc(const Dev& d, const void* tab, int tcm, int L, size_t smem, int grid, int nbuf, cudaStream_t s);

// the Gaunt coefficients into the constant memory of the module that holds the
// float expensive kernels of tcm and n_rad, on the current device
cudaError_t ace_gaunt_upload(int tcm, int n_rad, const float* g, int n);

// tensor-core building block check (k_tc.cu)
cudaError_t tc_selftest(const uint16_t* a, const uint16_t* b, int m, int n, int k, float* d, int* status,
                        cudaStream_t s);

// cheap potential (k_spline.cu)
// lpa: lanes per evaluated atom (32, or 16 or 8 for atoms with few neighbours);
// spline_nb3(lpa): three-body neighbours an atom may have on chip with lpa lanes
cudaError_t spline_configure(int precision, int lpa, size_t* smem, int* grid);
int spline_nb3(int lpa);
void launch_spline(const Dev& d, const void* tab, int precision, int lpa, size_t smem, int grid, cudaStream_t s);

// gather + blend + second half-kick (k_gather.cu)
void launch_gather(const Dev& d, int precision, int integrate, double h, cudaStream_t s);

// ---------------------------------------------------------------------------
// multi-system step (batches of contexts sharing one stream)

constexpr int GB_ATOMS = 8, GB_ATOMS_BIG = 32;   // atoms a warp of the batched gather (BatchPlan::gather_atoms)

// Block-table classes: every batched launch uses the table of its granularity.
enum BatchTabClass : int {
    BT_FRONT = 0,  // FRONT_ATOMS atoms (front)
    BT_GATHER,     // 8 warps of gather_atoms atoms each (gather)
    BT_COUNT
};

struct FlatArgs {
    const Dev* devs;
    int nsys;
    int ngrp;
    const int* egroup;   // [nsys] expensive group (systems sharing T, L, NP)
    const int* elast;    // [nsys] 1 for the last system of its group
    const int* ebase;    // [ngrp] start of each group in list_e
    int2* list_e;        // {system, first index of a group of ACE_GROUP in its expensive list}
    int2* list_c;        // {system, atom} for each entry of the systems' cheap lists
    int* counts;         // [ngrp + 1] expensive totals per group, cheap total
};

struct BatchPlan {
    BatchArgs ba[BT_COUNT];
    int nblk[BT_COUNT];
    const Regions* regions;   // [nsys]
    const double* hk;         // [nsys] half-kick factors of the plan's time step
    int* any;                 // set while some system rebuilds its lists in this step
    int gather_atoms;         // GB_ATOMS or GB_ATOMS_BIG
    int capp2;                // largest power-of-two list capacity (build scratch)
    FlatArgs flat;
};

// displacement, lists, weights, sets and their flattened lists of every system, a
// kernel a phase (k_front.cu)
int front_batch_kernels();
cudaError_t launch_front_batch(const BatchPlan& p, cudaStream_t s, int integrate, double dt);
cudaError_t ace_batch_configure(int precision, int L, int n, int cap, int tile_max, int qb, size_t* smem, int* grid);
void launch_ace_batch(int precision, const Dev* devs, const void* tabs, const int2* list, const int* count,
                      int n, int L, size_t smem, int grid, cudaStream_t s);
cudaError_t spline_batch_configure(int precision, int lpa, size_t* smem, int* grid);
void launch_spline_batch(int precision, int lpa, const Dev* devs, const void* tabs, const int2* list,
                         const int* count, int uniform, size_t smem, int grid, cudaStream_t s);
void launch_gather_batch(const BatchPlan& p, int precision, int integrate, cudaStream_t s);

int sm_count();

// Raise (never lower) a kernel's dynamic shared-memory limit to `bytes`.  The
// limit belongs to the kernel, not to a context: contexts of different sizes
// share kernel instantiations, so one context must not shrink another's limit.
cudaError_t raise_smem_limit(const void* func, size_t bytes);

// FMA throughput microbenchmark (k_peak.cu)
int fma_peak(int precision, cudaStream_t s, double* flops_per_s);

}  // namespace mixd
