// Multi-system (batched) kernels of the weights and sets (bodies in k_sets.cuh)
// and the ordered compaction of the evaluated sets into ascending index lists.
#include "k_sets.cuh"

namespace mixd {

constexpr int BUF_WARPS = 8;

// Per-block counts of the two evaluated sets (and of the diagnostic sets).
__device__ __forceinline__ void count_body(const Dev& d, int bx) {
    const int64_t i = bx * (int64_t)SCAN_BLOCK + threadIdx.x;
    int f = 0;
    double lam = 0.0;
    if (i < d.n) {
        f = d.flags[i];
        lam = d.lam[i];
    }
    const bool in = i < d.n;
    const int ne = __syncthreads_count(in && (f & 4));
    const int ncheap = __syncthreads_count(in && (f & 8));
    const int ncore = __syncthreads_count(in && lam == 1.0);
    const int nramp = __syncthreads_count(in && lam > 0.0 && lam < 1.0);
    const int nle = __syncthreads_count(in && (f & 1));
    const int nlc = __syncthreads_count(in && (f & 2));
    if (threadIdx.x == 0) {
        d.blk_e[bx] = ne;
        d.blk_c[bx] = ncheap;
        atomicAdd(d.status + SW_NCORE, ncore);
        atomicAdd(d.status + SW_NRAMP, nramp);
        atomicAdd(d.status + SW_NLE, nle);
        atomicAdd(d.status + SW_NLC, nlc);
    }
}

// Ordered compaction: act lists ascending, pos maps (-1 when not evaluated).
__device__ __forceinline__ void scatter_body(const Dev& d, int bx, int gx) {
    __shared__ int red_e[32], red_c[32];
    __shared__ int off_e_s, off_c_s;
    const int tid = threadIdx.x, lane = tid & 31, warp = tid >> 5;
    const int b = bx;
    // offset of this block: sum of the counts of the blocks before it
    int se = 0, sc = 0;
    for (int k = tid; k < b; k += SCAN_BLOCK) {
        se += d.blk_e[k];
        sc += d.blk_c[k];
    }
    for (int o = 16; o > 0; o >>= 1) {
        se += __shfl_down_sync(0xffffffffu, se, o);
        sc += __shfl_down_sync(0xffffffffu, sc, o);
    }
    if (lane == 0) {
        red_e[warp] = se;
        red_c[warp] = sc;
    }
    __syncthreads();
    if (warp == 0) {
        int a = red_e[lane], c = red_c[lane];
        for (int o = 16; o > 0; o >>= 1) {
            a += __shfl_down_sync(0xffffffffu, a, o);
            c += __shfl_down_sync(0xffffffffu, c, o);
        }
        if (lane == 0) {
            off_e_s = a;
            off_c_s = c;
        }
    }
    __syncthreads();
    const int64_t i = (int64_t)b * SCAN_BLOCK + tid;
    const int f = i < d.n ? d.flags[i] : 0;
    const bool ie = (f & 4) != 0, ic = (f & 8) != 0;
    const unsigned be = __ballot_sync(0xffffffffu, ie), bc = __ballot_sync(0xffffffffu, ic);
    const unsigned lt = (1u << lane) - 1u;
    __syncthreads();
    if (lane == 0) {
        red_e[warp] = __popc(be);
        red_c[warp] = __popc(bc);
    }
    __syncthreads();
    if (warp == 0) {
        int a = red_e[lane], c = red_c[lane];
        int ia = a, ic2 = c;
        for (int o = 1; o < 32; o <<= 1) {
            int ta = __shfl_up_sync(0xffffffffu, ia, o);
            int tc = __shfl_up_sync(0xffffffffu, ic2, o);
            if (lane >= o) {
                ia += ta;
                ic2 += tc;
            }
        }
        red_e[lane] = ia - a;   // exclusive per-warp offsets
        red_c[lane] = ic2 - c;
        if (lane == 31 && b == gx - 1) {
            d.status[SW_NEXP] = off_e_s + ia;
            d.status[SW_NCHEAP] = off_c_s + ic2;
        }
    }
    __syncthreads();
    if (i < d.n) {
        if (ie) {
            const int p = off_e_s + red_e[warp] + __popc(be & lt);
            d.act_e[p] = (int)i;
            d.pos_e[i] = p;
        } else {
            d.pos_e[i] = -1;
        }
        if (ic) {
            const int p = off_c_s + red_c[warp] + __popc(bc & lt);
            d.act_c[p] = (int)i;
            d.pos_c[i] = p;
        } else {
            d.pos_c[i] = -1;
        }
    }
}

// ---------------------------------------------------------------------------
// multi-system versions (geometric regions only)

__global__ void kb_lambda(BatchArgs ba, const Regions* __restrict__ regions) {
    MIX_BATCH_BLOCK(ba)
    __shared__ Regions s_reg;   // the system's regions, read per atom
    copy_shared(&s_reg, regions + s_ent.x);
    __syncthreads();
    lambda_body(s_dev, s_reg, s_ent.y, s_ent.z);
}
__global__ void __launch_bounds__(BUF_WARPS * 32) kb_buffer(BatchArgs ba) {
    MIX_BATCH_BLOCK(ba)
    buffer_dispatch(s_dev, s_ent.y, s_ent.z, 32);
}
__global__ void __launch_bounds__(SCAN_BLOCK) kb_count(BatchArgs ba) {
    MIX_BATCH_BLOCK(ba)
    count_body(s_dev, s_ent.y);
}
__global__ void __launch_bounds__(SCAN_BLOCK) kb_scatter(BatchArgs ba) {
    MIX_BATCH_BLOCK(ba)
    scatter_body(s_dev, s_ent.y, s_ent.z);
}

// Flattened lists of the evaluated atoms of every system: block s writes
// {s, i} for each atom i of its cheap list, and {s, ACE_GROUP k} for each group of
// ACE_GROUP consecutive atoms of its expensive list (a CTA of the expensive
// kernel takes one such group), at the sum of the counts of the systems before
// it (within its expensive group; all systems for cheap).  The last system of
// a group writes the group's total; the last system the cheap total.
__global__ void kb_flatten(FlatArgs f) {
    __shared__ int red[2][32];
    const int s = blockIdx.x, tid = threadIdx.x, lane = tid & 31, warp = tid >> 5;
    const int g = f.egroup[s];
    int oe = 0, oc = 0;
    for (int t = tid; t < s; t += blockDim.x) {
        const int* st = f.devs[t].status;
        if (f.egroup[t] == g) oe += (st[SW_NEXP] + ACE_GROUP - 1) / ACE_GROUP;
        oc += st[SW_NCHEAP];
    }
    for (int o = 16; o > 0; o >>= 1) {
        oe += __shfl_down_sync(0xffffffffu, oe, o);
        oc += __shfl_down_sync(0xffffffffu, oc, o);
    }
    if (lane == 0) {
        red[0][warp] = oe;
        red[1][warp] = oc;
    }
    __syncthreads();
    oe = 0;
    oc = 0;
    for (int w = 0; w < (int)(blockDim.x >> 5); ++w) {
        oe += red[0][w];
        oc += red[1][w];
    }
    const int* st = f.devs[s].status;
    const int ne = (st[SW_NEXP] + ACE_GROUP - 1) / ACE_GROUP, nc = st[SW_NCHEAP];
    int2* le = f.list_e + f.ebase[g] + oe;
    int2* lc = f.list_c + oc;
    for (int k = tid; k < ne; k += blockDim.x) le[k] = make_int2(s, k * ACE_GROUP);
    const int* act_c = f.devs[s].act_c;
    for (int k0 = tid; k0 < nc; k0 += 4 * blockDim.x) {   // four reads in flight a thread
        int v[4];
#pragma unroll
        for (int u = 0; u < 4; ++u)
            if (k0 + u * (int)blockDim.x < nc) v[u] = act_c[k0 + u * blockDim.x];
#pragma unroll
        for (int u = 0; u < 4; ++u)
            if (k0 + u * (int)blockDim.x < nc) lc[k0 + u * blockDim.x] = make_int2(s, v[u]);
    }
    if (tid == 0) {
        if (f.elast[s]) f.counts[g] = oe + ne;
        if (s == f.nsys - 1) f.counts[f.ngrp] = oc + nc;
    }
}

void launch_sets_batch(const BatchPlan& p, cudaStream_t s) {
    kb_lambda<<<p.nblk[BT_ATOM], 256, 0, s>>>(p.ba[BT_ATOM], p.regions);
    kb_buffer<<<p.nblk[BT_WARP8], BUF_WARPS * 32, 0, s>>>(p.ba[BT_WARP8]);
    kb_count<<<p.nblk[BT_SCAN], SCAN_BLOCK, 0, s>>>(p.ba[BT_SCAN]);
    kb_scatter<<<p.nblk[BT_SCAN], SCAN_BLOCK, 0, s>>>(p.ba[BT_SCAN]);
    kb_flatten<<<p.flat.nsys, 1024, 0, s>>>(p.flat);
}

}  // namespace mixd
