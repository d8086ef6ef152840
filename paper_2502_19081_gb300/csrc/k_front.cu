// The front of one evaluation in a single cooperative launch: first half-kick,
// drift and skin test, the lists when they are rebuilt, the blend weights, and
// the evaluated sets with their compaction.
//
// What bounds it: in a small system nothing but latency.  As ten kernels
// (displacement, five list kernels that mostly return at once, weights, buffer,
// counts, compaction) it took 2-7 us a kernel; here a step without a rebuild
// crosses the grid twice (three times beyond FRONT_REDUNDANT atoms, some 1.1 us
// each) and a rebuild is a branch.  Measured, steps without a rebuild: 8,001 atoms
// 15.7 us in all (as ten kernels 55 by their events), 1,000 atoms 11.4 (40),
// 200,000 atoms 54 (79).  The phases are separated by grid barriers, so the launch
// is cooperative (all CTAs resident, at most FRONT_CTAS an SM); every wait is
// bounded.  The price: two CTAs fill an SM's registers, so contexts on streams of
// their own no longer overlap their small kernels (24 silicon systems of 5,831 atoms,
// us a step and system: 39, as ten kernels 20; 8 iron dumbbells 116, as ten kernels
// 151).  One CTA an SM brought the first to 27 and cost a system alone up to 5 %;
// systems stepped together belong in a batch (15.8), whose front has kernels of
// its own.
#include <algorithm>
#include <map>
#include <mutex>
#include <utility>

#include "k_lists.cuh"
#include "k_sets.cuh"

namespace mixd {

namespace {

constexpr int FRONT_THREADS = 512;
constexpr int FRONT_WARPS = FRONT_THREADS / 32;
constexpr int FRONT_CTAS = 2;   // resident CTAs an SM the kernel is compiled for
// Up to this many atoms (cells) every CTA counts the flags (cell counts) before
// its own chunk itself, at most 32 KB from L2, instead of publishing its count
// and crossing the grid once more.
constexpr int FRONT_REDUNDANT = 32768;
constexpr int FRONT_REDUNDANT_CELLS = 8192;
struct FrontOpt {
    int integrate, force_rebuild;
    double dt, h;
    int capp2, tiled;
    int prof;              // write SW_CLOCK
    const double4* x_in;   // lists alone (mix_neighbours_noalloc): positions to copy; else null
};

__device__ __forceinline__ int ld_acquire(const int* p) {
    int v;
    asm volatile("ld.acquire.gpu.global.b32 %0, [%1];" : "=r"(v) : "l"(p) : "memory");
    return v;
}

// Every CTA of the grid arrives before any goes on.  The count only grows during
// a launch (a CTA's k-th barrier waits for k times the grid), which keeps a
// barrier at one reduction and one poll; the last CTA to leave the kernel clears
// it (done).  False once the wait gave up: then every thread of the CTA leaves, the
// status bit stays, and every later kernel of the context does nothing (list_ok).
struct Grid {
    int* status;
    int target, limit;   // limit: polls before a wait gives up
    __device__ __forceinline__ Grid(int* s, int polls) : status(s), target(0), limit(polls) {}
    __device__ __forceinline__ bool barrier() {
        __shared__ int s_ok;
        target += (int)gridDim.x;
        __syncthreads();
        if (threadIdx.x == 0) {
            asm volatile("red.release.gpu.global.add.s32 [%0], 1;" ::"l"(status + SW_GRID_COUNT) : "memory");
            int polls = 0;
            while (ld_acquire(status + SW_GRID_COUNT) < target && ++polls < limit) {
            }
            if (polls >= limit) set_status(status, ST_GRID_TIMEOUT);
            s_ok = polls < limit;
        }
        __syncthreads();
        return s_ok != 0;
    }
    __device__ __forceinline__ void done() {
        if (threadIdx.x == 0 && atomicAdd(status + SW_GRID_DONE, 1) == (int)gridDim.x - 1) {
            status[SW_GRID_COUNT] = 0;
            status[SW_GRID_DONE] = 0;
        }
    }
};

// Calls f(i) for every atom, 32 consecutive atoms a warp, the warps' shares dealt
// out CTA by CTA: a small system's atoms land on as many SMs as there are CTAs.  A
// warp-wide float64 instruction holds an SM's float64 pipe for 16 cycles, so 16
// warps of one CTA side by side take 17 us for the displacement and the weights
// where one warp takes one (1,000 atoms: 2 CTAs of 512 against 32 of 32).
template <class F>
__device__ __forceinline__ void for_atoms(int64_t n, F&& f) {
    const int lane = threadIdx.x & 31, warp = threadIdx.x >> 5;
    const int64_t gx = gridDim.x;
    for (int64_t c = warp * gx + blockIdx.x; c * 32 < n; c += FRONT_WARPS * gx) {
        const int64_t i = c * 32 + lane;
        if (i < n) f(i);
    }
}

// exclusive offset of this thread's value within the CTA, and the CTA's total
__device__ __forceinline__ int2 block_scan2(int a, int b, int2* total) {
    __shared__ int2 ws[FRONT_WARPS];
    const int lane = threadIdx.x & 31, warp = threadIdx.x >> 5;
    int ia = a, ib = b;
#pragma unroll
    for (int o = 1; o < 32; o <<= 1) {
        const int ta = __shfl_up_sync(0xffffffffu, ia, o), tb = __shfl_up_sync(0xffffffffu, ib, o);
        if (lane >= o) {
            ia += ta;
            ib += tb;
        }
    }
    __syncthreads();   // the previous use of ws is over
    if (lane == 31) ws[warp] = make_int2(ia, ib);
    __syncthreads();
    int pa = 0, pb = 0, ta = 0, tb = 0;
#pragma unroll
    for (int w = 0; w < FRONT_WARPS; ++w) {
        const int2 v = ws[w];
        if (w < warp) {
            pa += v.x;
            pb += v.y;
        }
        ta += v.x;
        tb += v.y;
    }
    *total = make_int2(ta, tb);
    return make_int2(pa + ia - a, pb + ib - b);
}

__device__ __forceinline__ int2 block_sum2(int a, int b) {
    int2 t;
    block_scan2(a, b, &t);
    return t;
}

// Exclusive scan of the cell counts, a chunk of cells per CTA.  Returns false when
// a barrier gave up.  The counts are cleared by the fill phase's successor.
__device__ __forceinline__ bool front_cell_scan(const Dev& d, Grid& grid) {
    const int nc = d.cells.ncell, gx = (int)gridDim.x, bx = (int)blockIdx.x;
    const int chunk = (nc + gx - 1) / gx, c0 = min(bx * chunk, nc), c1 = min(c0 + chunk, nc);
    int before = 0;
    if (nc <= FRONT_REDUNDANT_CELLS) {
        int v = 0;
        for (int k = threadIdx.x; k < c0; k += FRONT_THREADS) v += d.cell_count[k];
        before = block_sum2(v, 0).x;
    } else {
        int v = 0;
        for (int k = c0 + threadIdx.x; k < c1; k += FRONT_THREADS) v += d.cell_count[k];
        const int own = block_sum2(v, 0).x;
        if (threadIdx.x == 0) d.blk_e[bx] = own;
        if (!grid.barrier()) return false;
        v = 0;
        for (int k = threadIdx.x; k < bx; k += FRONT_THREADS) v += d.blk_e[k];
        before = block_sum2(v, 0).x;
    }
    for (int base = c0; base < c1; base += FRONT_THREADS) {
        const int k = base + (int)threadIdx.x;
        const int v = k < c1 ? d.cell_count[k] : 0;
        int2 tot;
        const int ex = before + block_scan2(v, 0, &tot).x;
        if (k < c1) {
            d.cell_start[k] = ex;
            d.cell_fill[k] = 0;
        }
        before += tot.x;
    }
    if (bx == gx - 1 && threadIdx.x == 0) d.cell_start[nc] = before;
    if (bx == 0 && threadIdx.x == 0) d.status[SW_MAXNB] = 0;
    return true;
}

// The lists of the current positions (the phases of the batched list kernels)
__device__ __forceinline__ bool front_build(const Dev& d, Grid& grid, int capp2, int tiled, unsigned char* smem) {
    const int bx = (int)blockIdx.x, gx = (int)gridDim.x;
    for_atoms(d.n, [&](int64_t i) { cell_bin_atom(d, i); });
    if (!grid.barrier()) return false;
    if (!front_cell_scan(d, grid)) return false;
    if (!grid.barrier()) return false;
    cell_fill_body(d, bx, gx);
    if (!grid.barrier()) return false;
    for (int k = bx * FRONT_THREADS + threadIdx.x; k < d.cells.ncell; k += gx * FRONT_THREADS) d.cell_count[k] = 0;
    if (tiled) neigh_build_tiled_body<FRONT_WARPS>(d, bx, gx, capp2, smem);
    else neigh_build_body<FRONT_WARPS>(d, bx, gx, capp2, reinterpret_cast<int*>(smem));
    if (!grid.barrier()) return false;
    neigh_rev_body(d, bx, gx);
    return true;
}

// Ordered compaction of the evaluated sets: CTA b takes the b-th chunk of atoms.
__device__ __forceinline__ bool front_compact(const Dev& d, Grid& grid) {
    const int gx = (int)gridDim.x, bx = (int)blockIdx.x, n = (int)d.n;
    const int chunk = ((n + gx - 1) / gx + 31) & ~31, a0 = min(bx * chunk, n), a1 = min(a0 + chunk, n);
    int2 before;
    if (n <= FRONT_REDUNDANT) {
        // flags bits 2 and 3 (expensive, cheap), sixteen atoms a load (a0 is a
        // multiple of 32, except where the chunk is empty and nothing is written)
        int se = 0, sc = 0;
        const uint4* w = reinterpret_cast<const uint4*>(d.flags);
        const int full = a0 < n ? a0 / 16 : 0;
        for (int k = threadIdx.x; k < full; k += FRONT_THREADS) {
            const uint4 v = w[k];
            se += __popc(v.x & 0x04040404u) + __popc(v.y & 0x04040404u) + __popc(v.z & 0x04040404u) + __popc(v.w & 0x04040404u);
            sc += __popc(v.x & 0x08080808u) + __popc(v.y & 0x08080808u) + __popc(v.z & 0x08080808u) + __popc(v.w & 0x08080808u);
        }
        before = block_sum2(se, sc);
    } else {
        int se = 0, sc = 0;
        for (int i = a0 + threadIdx.x; i < a1; i += FRONT_THREADS) {
            const int f = d.flags[i];
            se += (f >> 2) & 1;
            sc += (f >> 3) & 1;
        }
        const int2 own = block_sum2(se, sc);
        if (threadIdx.x == 0) {
            d.blk_e[bx] = own.x;
            d.blk_c[bx] = own.y;
        }
        if (!grid.barrier()) return false;
        se = sc = 0;
        for (int k = threadIdx.x; k < bx; k += FRONT_THREADS) {
            se += d.blk_e[k];
            sc += d.blk_c[k];
        }
        before = block_sum2(se, sc);
    }
    int ncore = 0, nramp = 0, nle = 0, nlc = 0;
    for (int base = a0; base < a1; base += FRONT_THREADS) {
        const int i = base + (int)threadIdx.x;
        const bool in = i < a1;
        const int f = in ? d.flags[i] : 0;
        const double lam = in ? d.lam[i] : 0.0;
        const int ie = (f >> 2) & 1, ic = (f >> 3) & 1;
        int2 tot;
        const int2 ex = block_scan2(ie, ic, &tot);
        if (in) {
            const int pe = before.x + ex.x, pc = before.y + ex.y;
            if (ie) d.act_e[pe] = i;
            if (ic) d.act_c[pc] = i;
            d.pos_e[i] = ie ? pe : -1;
            d.pos_c[i] = ic ? pc : -1;
        }
        before.x += tot.x;
        before.y += tot.y;
        // the CTA's counts (__syncthreads_count would count every thread; a ballot
        // a warp and one atomic a warp below)
        ncore += __popc(__ballot_sync(0xffffffffu, in && lam == 1.0));
        nramp += __popc(__ballot_sync(0xffffffffu, in && lam > 0.0 && lam < 1.0));
        nle += __popc(__ballot_sync(0xffffffffu, (f & 1) != 0));
        nlc += __popc(__ballot_sync(0xffffffffu, (f & 2) != 0));
    }
    if ((threadIdx.x & 31) == 0) {
        if (ncore) atomicAdd(d.status + SW_NCORE, ncore);
        if (nramp) atomicAdd(d.status + SW_NRAMP, nramp);
        if (nle) atomicAdd(d.status + SW_NLE, nle);
        if (nlc) atomicAdd(d.status + SW_NLC, nlc);
    }
    // the CTA that holds the last atom (chunks are rounded up: later CTAs are empty)
    if (a1 == n && (a0 < n || bx == 0) && threadIdx.x == 0) {
        d.status[SW_NEXP] = before.x;
        d.status[SW_NCHEAP] = before.y;
    }
    return true;
}

__device__ __forceinline__ void front_lambda(const Dev& d, const Regions& r) {
    for_atoms(d.n, [&](int64_t i) { lambda_atom(d, r, i); });
}

__global__ void __launch_bounds__(FRONT_THREADS, FRONT_CTAS) k_front(Dev d, Regions r, SeedRule sr, FrontOpt o, int apw) {
    extern __shared__ __align__(16) unsigned char front_smem[];
    if (!list_ok(d)) return;
    Grid grid(d.status, d.grid_polls);
    const int bx = (int)blockIdx.x, gx = (int)gridDim.x;
    const bool g0 = bx == 0 && threadIdx.x == 0;
    // a phase ends (k = 1: displacement, 2: lists, 3: sets) as this CTA sees it
    auto stamp = [&](int k) {
        if (o.prof && g0) reinterpret_cast<long long*>(d.status + SW_CLOCK)[k] = clock64();
    };
    stamp(0);
    if (g0) disp_reset(d, o.force_rebuild);
    // displacement, and the weights of the drifted positions at once: they stand
    // unless the lists are rebuilt (which folds the positions)
    for_atoms(d.n, [&](int64_t i) {
        disp_atom(d, i, o.integrate, o.dt, o.h, o.force_rebuild);
        if (sr.mode == 0 && !o.force_rebuild) lambda_atom(d, r, i);
    });
    if (!grid.barrier()) return;
    stamp(1);
    const bool rebuild = o.force_rebuild || ld_acquire(d.status + SW_REBUILD) != 0;
    if (rebuild) {
        if (!front_build(d, grid, o.capp2, o.tiled, front_smem)) return;
        if (sr.mode == 0) front_lambda(d, r);
        if (!grid.barrier()) return;
        if (g0) {   // every CTA has read the flag
            d.status[SW_REBUILDS] += 1;
            d.status[SW_REBUILD] = 0;
        }
        stamp(2);
    }
    if (sr.mode != 0) {
        if (sr.mode == 2) {
            coord_body(d, sr, bx, gx);
            if (!grid.barrier()) return;
        }
        core_body(d, sr, bx, gx);
        if (!grid.barrier()) return;
        blend_body(d, sr, bx, gx);
        if (!grid.barrier()) return;
    }
    buffer_dispatch(d, bx, gx, apw);
    if (!grid.barrier()) return;
    if (front_compact(d, grid)) {
        if (!rebuild && o.prof && g0) {   // no lists
            const volatile long long* t = reinterpret_cast<const long long*>(d.status + SW_CLOCK);
            reinterpret_cast<long long*>(d.status + SW_CLOCK)[2] = t[1];
        }
        stamp(3);
        grid.done();
    }
}

// lists alone: positions copied and checked, counts cleared, then the build
__global__ void __launch_bounds__(FRONT_THREADS, FRONT_CTAS) k_front_lists(Dev d, FrontOpt o) {
    extern __shared__ __align__(16) unsigned char front_smem[];
    Grid grid(d.status, d.grid_polls);
    const int64_t g0 = (int64_t)blockIdx.x * FRONT_THREADS + threadIdx.x, gs = (int64_t)gridDim.x * FRONT_THREADS;
    for (int64_t k = g0; k < d.cells.ncell; k += gs) d.cell_count[k] = 0;
    for_atoms(d.n, [&](int64_t i) {
        const double4 x = o.x_in[i];
        d.x[i] = x;
        if (!(isfinite(x.x) && isfinite(x.y) && isfinite(x.z))) {
            set_status(d.status, ST_NONFINITE);
            return;
        }
        const double xs[3] = {x.x, x.y, x.z};
        for (int k = 0; k < 3; ++k)
            if (!d.box.per[k] && (xs[k] < d.box.lo[k] || xs[k] >= d.box.lo[k] + d.box.L[k]))
                set_status(d.status, ST_OUT_OF_BOX);
    });
    if (!grid.barrier()) return;
    if (front_build(d, grid, o.capp2, o.tiled, front_smem)) grid.done();
}

// The front of every system of a batch: the phases of k_front as kernels of their
// own.  The work comes in table entries of FRONT_ATOMS consecutive atoms of one
// system (a thread each), a block an entry with the entry's system in shared
// memory.  The bodies are those of k_front, so a system's lists and sets are the
// ones it gets alone; the list phases return at once when no system needs them and
// for the systems that do not; the compaction also writes the flattened lists the
// batched potentials walk.
// One cooperative launch for all phases, as for a single system, loses here: its 64
// registers and 32 warps an SM hold in every phase, and in a batch some member
// rebuilds in most steps, with its few entries on as many blocks.  Steps at 50 K,
// 20 at a time, one kernel / eight, us: 2 systems of 1,000 silicon atoms 112 / 90, 8
// of them 187 / 124, 24 of them 305 / 186, 11 of 5,831 atoms 294 / 219, 8 iron
// systems of 1,023 atoms 424 / 322, 8 of 8,191 atoms 1,034 / 958; 256 of 5,831 silicon
// atoms with every member rebuilding 5.9 / 1.9 ms for the front alone.
struct FrontBatch {
    BatchPlan p;
    int integrate;
    double dt;
};

enum { FB_DISP, FB_BIN, FB_SCAN, FB_FILL, FB_ROWS, FB_REV, FB_BUFFER, FB_LISTS, FB_COUNT };

// list rows in blocks of 4 warps, so that a system that rebuilds is spread over many SMs
__host__ __device__ constexpr int fb_threads(int ph) { return ph == FB_ROWS ? 128 : (ph == FB_REV ? 256 : FRONT_THREADS); }
__host__ __device__ constexpr int fb_blocks(int ph) { return ph == FB_ROWS ? 16 : (ph == FB_REV ? 4 : 1); }   // blocks an entry

__device__ __forceinline__ void front_batch_disp(const FrontBatch& f, const int4& e, const Dev& d, const Regions& r) {
    const int64_t i = (int64_t)e.y * FRONT_ATOMS + threadIdx.x;
    if (e.y == 0 && threadIdx.x == 0) {
        disp_reset(d, 0);
        d.status[SW_NEXP] = 0;
        d.status[SW_NCHEAP] = 0;
    }
    if (list_ok(d) && i < d.n) {
        if (disp_atom(d, i, f.integrate, f.dt, f.p.hk[e.x], 0)) *f.p.any = 1;
        lambda_atom(d, r, i);   // stands unless the lists are rebuilt
    }
}

// buffers; a warp's 32 atoms are its own, so it counts them at once
__device__ __forceinline__ void front_batch_buffer(const BatchPlan& p, const int4& e, const Dev& d) {
    const int lane = threadIdx.x & 31;
    const bool ok = list_ok(d);
    if (ok) buffer_dispatch(d, e.y, e.z, 32);
    const int64_t i = (int64_t)e.y * FRONT_ATOMS + threadIdx.x;
    const bool in = ok && i < d.n;
    const int fl = in ? d.flags[i] : 0;
    const double lam = in ? d.lam[i] : 0.0;
    const int2 own = block_sum2((fl >> 2) & 1, (fl >> 3) & 1);
    if (threadIdx.x == 0) {
        d.blk_e[e.y] = own.x;
        d.blk_c[e.y] = own.y;
        if (own.x) atomicAdd(d.status + SW_NEXP, own.x);
        if (own.y) atomicAdd(d.status + SW_NCHEAP, own.y);
        if (ok && e.y == 0 && d.status[SW_REBUILD]) {
            d.status[SW_REBUILDS] += 1;
            d.status[SW_REBUILD] = 0;
        }
        if (blockIdx.x == 0) *p.any = 0;   // the list phases are over
    }
    const int ncore = __popc(__ballot_sync(0xffffffffu, in && lam == 1.0));
    const int nramp = __popc(__ballot_sync(0xffffffffu, in && lam > 0.0 && lam < 1.0));
    const int nle = __popc(__ballot_sync(0xffffffffu, (fl & 1) != 0));
    const int nlc = __popc(__ballot_sync(0xffffffffu, (fl & 2) != 0));
    if (lane == 0) {
        if (ncore) atomicAdd(d.status + SW_NCORE, ncore);
        if (nramp) atomicAdd(d.status + SW_NRAMP, nramp);
        if (nle) atomicAdd(d.status + SW_NLE, nle);
        if (nlc) atomicAdd(d.status + SW_NLC, nlc);
    }
}

__device__ __forceinline__ void front_batch_lists(const BatchPlan& p, const int4& e, const Dev& d) {
    const FlatArgs& fa = p.flat;
    const int s = e.x;
    // this entry's place in its system's lists, and the system's in the flattened ones
    int se = 0, sc = 0, oe = 0, oc = 0;
    for (int t = threadIdx.x; t < e.y; t += FRONT_THREADS) {
        se += d.blk_e[t];
        sc += d.blk_c[t];
    }
    const int g = fa.egroup[s];
    for (int t = threadIdx.x; t < s; t += FRONT_THREADS) {
        const int* st = fa.devs[t].status;
        if (fa.egroup[t] == g) oe += (st[SW_NEXP] + ACE_GROUP - 1) / ACE_GROUP;
        oc += st[SW_NCHEAP];
    }
    const int2 before = block_sum2(se, sc), flat = block_sum2(oe, oc);
    const int64_t i = (int64_t)e.y * FRONT_ATOMS + threadIdx.x;
    const bool in = list_ok(d) && i < d.n;
    const int fl = in ? d.flags[i] : 0;
    const int ie = (fl >> 2) & 1, ic = (fl >> 3) & 1;
    int2 tot;
    const int2 ex = block_scan2(ie, ic, &tot);
    if (in) {
        const int pe = before.x + ex.x, pc = before.y + ex.y;
        if (ie) d.act_e[pe] = (int)i;
        if (ic) {
            d.act_c[pc] = (int)i;
            fa.list_c[flat.y + pc] = make_int2(s, (int)i);
        }
        d.pos_e[i] = ie ? pe : -1;
        d.pos_c[i] = ic ? pc : -1;
    }
    if (e.y == 0) {
        const int ne = (d.status[SW_NEXP] + ACE_GROUP - 1) / ACE_GROUP, nc = d.status[SW_NCHEAP];
        int2* le = fa.list_e + fa.ebase[g] + flat.x;
        for (int t = threadIdx.x; t < ne; t += FRONT_THREADS) le[t] = make_int2(s, t * ACE_GROUP);
        if (threadIdx.x == 0) {
            if (fa.elast[s]) fa.counts[g] = flat.x + ne;
            if (s == fa.nsys - 1) fa.counts[fa.ngrp] = flat.y + nc;
        }
    }
}

// A member whose own front gave up at a barrier before it was stepped with the batch
// (list_ok) may have half-written lists: it takes no part, with empty sets, until it
// is bound again.  No kernel of a batch sets that bit, so a block reads one value.
template <int PH>
__global__ void __launch_bounds__(fb_threads(PH), PH == FB_ROWS ? 8 : (PH == FB_REV ? 1 : 2))
    kb_front_phase(const __grid_constant__ FrontBatch f) {
    extern __shared__ __align__(16) unsigned char front_smem[];
    __shared__ Dev d;
    __shared__ Regions r;
    const BatchPlan& p = f.p;
    constexpr bool LISTS = PH != FB_DISP && PH != FB_BUFFER && PH != FB_LISTS;   // a phase of the rebuild
    if (LISTS && !*p.any) return;
    // this block's share of the system, a block a system for the scan
    constexpr int NB = fb_blocks(PH);
    int4 e = make_int4(blockIdx.x, 0, 1, 0);
    if constexpr (PH != FB_SCAN) e = p.ba[BT_FRONT].tab[blockIdx.x / NB];
    if (LISTS && !p.flat.devs[e.x].status[SW_REBUILD]) return;   // the whole block
    if (LISTS && !list_ok(p.flat.devs[e.x].status)) return;
    load_dev(&d, p.flat.devs + e.x);
    if constexpr (PH == FB_DISP || PH == FB_BIN) copy_shared(&r, p.regions + e.x);
    __syncthreads();
    const int bx = e.y * NB + (int)(blockIdx.x % NB), gx = e.z * NB;
    if constexpr (PH == FB_DISP) {
        front_batch_disp(f, e, d, r);
    } else if constexpr (PH == FB_BUFFER) {
        front_batch_buffer(p, e, d);
    } else if constexpr (PH == FB_LISTS) {
        front_batch_lists(p, e, d);
    } else if constexpr (PH == FB_BIN) {
        const int64_t i = (int64_t)e.y * FRONT_ATOMS + threadIdx.x;
        if (i < d.n) {
            cell_bin_atom(d, i);
            lambda_atom(d, r, i);   // of the folded position
        }
    } else if constexpr (PH == FB_SCAN) {
        cell_scan_body(d);
    } else if constexpr (PH == FB_FILL) {
        cell_fill_body(d, bx, gx);
    } else if constexpr (PH == FB_ROWS) {
        neigh_build_body<fb_threads(FB_ROWS) / 32>(d, bx, gx, pow2_cap(d.cap), reinterpret_cast<int*>(front_smem));
    } else {
        neigh_rev_body(d, bx, gx);
    }
}

template <int PH>
cudaError_t launch_front_phase(const FrontBatch& f, int units, size_t smem, cudaStream_t s) {
    const cudaError_t e = raise_smem_limit((const void*)kb_front_phase<PH>, smem);
    if (e != cudaSuccess) return e;
    kb_front_phase<PH><<<units * fb_blocks(PH), fb_threads(PH), smem, s>>>(f);
    return cudaPeekAtLastError();
}

// CTAs that are resident together with `smem` bytes each (0 on an error)
int front_resident(const void* kern, size_t smem) {
    int per_sm = 0;
    if (raise_smem_limit(kern, smem) != cudaSuccess) return 0;
    if (cudaOccupancyMaxActiveBlocksPerMultiprocessor(&per_sm, kern, FRONT_THREADS, smem) != cudaSuccess) return 0;
    return std::min(per_sm * sm_count(), FRONT_MAX_CTAS);
}

// the same for the lists-only kernel, which has no context to keep it in: asked
// once per device and shape (the shared memory depends on the row capacity alone)
int lists_resident(size_t smem) {
    static std::mutex mu;
    static std::map<std::pair<int, size_t>, int> known;
    int dev = 0;
    if (cudaGetDevice(&dev) != cudaSuccess) return 0;
    std::lock_guard<std::mutex> lock(mu);
    auto it = known.find({dev, smem});
    if (it != known.end()) return it->second;
    const int n = front_resident((const void*)k_front_lists, smem);
    if (n > 0) known[{dev, smem}] = n;
    return n;
}

// Lists a cell at a time (candidates staged in shared memory, a team of warps a
// cell) or an atom at a time: the first where the cells fill the resident teams,
// the waves of cells at least three quarters full on the whole or more than four.  Some
// cells more than a wave leave most teams idle for its length.  Front of an
// evaluation that rebuilds, us, a cell / an atom at a time, 1,216 teams: iron, 343
// cells 111 / 80, 729 121 / 116, 1,000 122 / 129, 1,331 151 / 130, 1,584 166 / 165, 2,744
// 223 / 230; silicon,
// 512 cells 51 / 47, 1,000 55 / 56, 1,728 69 / 67, 2,548 82 / 82, 4,096 98 / 102.
bool front_tiled(const Dev& d) {
    if (!nb_tiled_ok(d)) return false;
    const int64_t teams = (int64_t)sm_count() * FRONT_CTAS * (FRONT_WARPS / NB_TEAM);
    const int64_t waves = (d.cells.ncell + teams - 1) / teams;
    return waves > 4 || 4 * (int64_t)d.cells.ncell >= 3 * waves * teams;
}

size_t front_shape(const Dev& d, FrontOpt& o) {
    o.capp2 = 32;
    while (o.capp2 < d.cap) o.capp2 <<= 1;
    o.tiled = front_tiled(d) ? 1 : 0;
    return o.tiled ? nb_tiled_smem(o.capp2, FRONT_WARPS) : (size_t)FRONT_WARPS * o.capp2 * sizeof(int);
}

}  // namespace

cudaError_t front_configure(Dev& d) {
    FrontOpt o{};
    const size_t smem = front_shape(d, o);
    d.grid_front_max = front_resident((const void*)k_front, smem);
    return d.grid_front_max > 0 ? cudaSuccess : cudaErrorInvalidConfiguration;
}

cudaError_t launch_front(const Dev& d, const Regions& r, const SeedRule& sr, cudaStream_t s, int integrate, double dt,
                         double h, int force_rebuild, bool prof) {
    FrontOpt o{};
    o.prof = prof ? 1 : 0;
    o.integrate = integrate;
    o.force_rebuild = force_rebuild;
    o.dt = dt;
    o.h = h;
    const size_t smem = front_shape(d, o);
    // a warp per atom in a small system (the buffer scans and list rows run side
    // by side), the resident CTAs in a large one
    const int64_t want = (d.n + FRONT_WARPS - 1) / FRONT_WARPS;
    int64_t lim = d.grid_front_max;
    if (d.grid_buffer > 0 && d.grid_buffer < lim) lim = d.grid_buffer;
    const int grid = (int)std::max<int64_t>(1, std::min(want, lim));
    // atoms per warp of the buffer scan: one up to 512 atoms per SM (a
    // 256,000-atom system gets 3, which keeps its shell of scanning atoms spread
    // over many warps), up to 32 beyond
    const int64_t warps_full = (int64_t)sm_count() * 512;
    int apw = (int)std::min<int64_t>(32, std::max<int64_t>(1, (d.n + warps_full - 1) / warps_full));
    Dev dd = d;
    Regions rr = r;
    SeedRule ss = sr;
    void* args[] = {&dd, &rr, &ss, &o, &apw};
    return cudaLaunchCooperativeKernel((const void*)k_front, dim3(grid), dim3(FRONT_THREADS), args, smem, s);
}

int front_batch_kernels() { return FB_COUNT; }

cudaError_t launch_front_batch(const BatchPlan& p, cudaStream_t s, int integrate, double dt) {
    static_assert(FRONT_ATOMS == FRONT_THREADS, "an entry's atoms are a block's threads");
    const FrontBatch f{p, integrate, dt};
    const int nent = p.nblk[BT_FRONT];
    const size_t rows = (size_t)(fb_threads(FB_ROWS) / 32) * p.capp2 * sizeof(int);
    cudaError_t e = launch_front_phase<FB_DISP>(f, nent, 0, s);
    if (e == cudaSuccess) e = launch_front_phase<FB_BIN>(f, nent, 0, s);
    if (e == cudaSuccess) e = launch_front_phase<FB_SCAN>(f, p.flat.nsys, 0, s);
    if (e == cudaSuccess) e = launch_front_phase<FB_FILL>(f, nent, 0, s);
    if (e == cudaSuccess) e = launch_front_phase<FB_ROWS>(f, nent, rows, s);
    if (e == cudaSuccess) e = launch_front_phase<FB_REV>(f, nent, 0, s);
    if (e == cudaSuccess) e = launch_front_phase<FB_BUFFER>(f, nent, 0, s);
    if (e == cudaSuccess) e = launch_front_phase<FB_LISTS>(f, nent, 0, s);
    return e;
}

cudaError_t launch_front_lists(const Dev& d, const double4* x_in, cudaStream_t s) {
    FrontOpt o{};
    const size_t smem = front_shape(d, o);
    o.x_in = x_in;
    const int64_t want = (d.n + FRONT_WARPS - 1) / FRONT_WARPS;
    const int lim = lists_resident(smem);
    if (lim < 1) return cudaErrorInvalidConfiguration;
    const int grid = (int)std::max<int64_t>(1, std::min<int64_t>(want, lim));
    Dev dd = d;
    void* args[] = {&dd, &o};
    return cudaLaunchCooperativeKernel((const void*)k_front_lists, dim3(grid), dim3(FRONT_THREADS), args, smem, s);
}

}  // namespace mixd
