// Multi-system (batched) kernels of the lists (bodies in k_lists.cuh) and small
// launch helpers.
#include <mutex>

#include "k_lists.cuh"

namespace mixd {

// ---------------------------------------------------------------------------
// multi-system versions (one launch for all systems of a batch)

__global__ void kb_disp(BatchArgs ba, int integrate, double dt, int force_rebuild) {
    MIX_BATCH_BLOCK(ba)
    disp_body(s_dev, s_ent.y, s_ent.z, integrate, dt, half_kick(dt, s_dev.mass), force_rebuild);
}
__global__ void kb_cell_bin(BatchArgs ba) {
    MIX_BATCH_BLOCK_REBUILD(ba)
    cell_bin_body(s_dev, s_ent.y, s_ent.z);
}
__global__ void kb_cell_scan(BatchArgs ba) {
    MIX_BATCH_BLOCK_REBUILD(ba)
    cell_scan_body(s_dev);
}
__global__ void kb_cell_fill(BatchArgs ba) {
    MIX_BATCH_BLOCK_REBUILD(ba)
    cell_fill_body(s_dev, s_ent.y, s_ent.z);
}
__global__ void __launch_bounds__(NB_WARPS * 32) kb_neigh_build(BatchArgs ba) {
    extern __shared__ __align__(16) int sbuf[];
    MIX_BATCH_BLOCK_REBUILD(ba)
    neigh_build_body<true, NB_WARPS>(s_dev, s_ent.y, s_ent.z, pow2_cap(s_dev.cap), sbuf);
}
__global__ void kb_neigh_rev(BatchArgs ba) {
    MIX_BATCH_BLOCK_REBUILD(ba)
    neigh_rev_body(s_dev, s_ent.y, s_ent.z);
}

static int g_sms = 0;

int sm_count() {
    if (g_sms == 0) {
        int dev = 0;
        cudaGetDevice(&dev);
        cudaDeviceGetAttribute(&g_sms, cudaDevAttrMultiProcessorCount, dev);
        if (g_sms <= 0) g_sms = 1;
    }
    return g_sms;
}

cudaError_t raise_smem_limit(const void* func, size_t bytes) {
    static std::mutex mu;
    std::lock_guard<std::mutex> lock(mu);
    cudaFuncAttributes fa;
    cudaError_t e = cudaFuncGetAttributes(&fa, func);
    if (e != cudaSuccess) return e;
    if ((size_t)fa.maxDynamicSharedSizeBytes >= bytes) return cudaSuccess;
    return cudaFuncSetAttribute(func, cudaFuncAttributeMaxDynamicSharedMemorySize, (int)bytes);
}

void launch_disp_batch(const BatchPlan& p, cudaStream_t s, int integrate, double dt, int force_rebuild) {
    kb_disp<<<p.nblk[BT_ATOM], 256, 0, s>>>(p.ba[BT_ATOM], integrate, dt, force_rebuild);
}

void launch_build_batch(const BatchPlan& p, cudaStream_t s) {
    kb_cell_bin<<<p.nblk[BT_ATOM], 256, 0, s>>>(p.ba[BT_ATOM]);
    kb_cell_scan<<<p.nblk[BT_ONE], 1024, 0, s>>>(p.ba[BT_ONE]);
    kb_cell_fill<<<p.nblk[BT_ATOM], 256, 0, s>>>(p.ba[BT_ATOM]);
    kb_neigh_build<<<p.nblk[BT_NB], NB_WARPS * 32, NB_WARPS * p.capp2 * sizeof(int), s>>>(p.ba[BT_NB]);
    kb_neigh_rev<<<p.nblk[BT_REV], 256, 0, s>>>(p.ba[BT_REV]);
}

}  // namespace mixd
