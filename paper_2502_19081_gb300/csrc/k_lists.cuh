// Device bodies: cell list and full neighbour list with a reverse-slot map (the region and
// force steps reuse one neighbour list, as the paper's region fix reuses the
// pair style's lists, Sec. 4.4), plus the first half of velocity Verlet and
// the skin test that decides when the lists are rebuilt.
//
// Bit-reproducibility: positions are folded, binned and compared with explicit
// round-to-nearest operations (no FMA), in the same order as a plain CPU
// evaluation: d = x_j - x_i; d -= L rint(d / L); r2 = dx*dx + dy*dy + dz*dz;
// neighbour iff r2 < (rc + skin)^2.  Each row of the list is sorted ascending.
#pragma once

#include <climits>

#include "mix_launch.h"

namespace mixd {

// The counters of one evaluation, reset by one thread.
__device__ __forceinline__ void disp_reset(const Dev& d, int force_rebuild) {
    d.status[SW_NCORE] = 0;
    d.status[SW_NRAMP] = 0;
    d.status[SW_NLE] = 0;
    d.status[SW_NLC] = 0;
    d.status[SW_EPOCH] += 1;
    if (force_rebuild) d.status[SW_REBUILD] = 1;
}

// v += h F; x += dt v (when integrating); then flag a rebuild if the atom moved
// more than skin/2 since the last build (returned as well).
__device__ __forceinline__ bool disp_atom(const Dev& d, int64_t i, int integrate, double dt, double h,
                                          int force_rebuild) {
    // every load first, so that one memory latency covers them all (the
    // arrays never overlap, which the compiler cannot know)
    double4 x = d.x[i];
    double4 v = make_double4(0.0, 0.0, 0.0, 0.0), f = v, xb = v;
    int c3 = 0;
    if (integrate) {
        v = d.v[i];
        f = d.f[i];
    }
    if (!force_rebuild) {
        xb = d.xb[i];
        if (d.xr) c3 = d.cell3[i];
    }
    if (integrate) {
        v.x = __dadd_rn(v.x, __dmul_rn(h, f.x));
        v.y = __dadd_rn(v.y, __dmul_rn(h, f.y));
        v.z = __dadd_rn(v.z, __dmul_rn(h, f.z));
        x.x = __dadd_rn(x.x, __dmul_rn(dt, v.x));
        x.y = __dadd_rn(x.y, __dmul_rn(dt, v.y));
        x.z = __dadd_rn(x.z, __dmul_rn(dt, v.z));
        d.v[i] = v;
        d.x[i] = x;
    }
    const bool finite = isfinite(x.x) && isfinite(x.y) && isfinite(x.z);
    if (!finite) {
        set_status(d.status, ST_NONFINITE);
        return false;
    }
    bool moved = false;
    const double xs[3] = {x.x, x.y, x.z};
    for (int k = 0; k < 3; ++k)
        if (!d.box.per[k] && (xs[k] < d.box.lo[k] || xs[k] >= d.box.lo[k] + d.box.L[k]))
            set_status(d.status, ST_OUT_OF_BOX);
    if (!force_rebuild) {
        const double dx = x.x - xb.x, dy = x.y - xb.y, dz = x.z - xb.z;
        moved = dx * dx + dy * dy + dz * dz > d.half_skin2;
        if (moved) d.status[SW_REBUILD] = 1;
        // relative to the cell of the last build (recomputed by the binning on rebuilds)
        if (d.xr) d.xr[i] = cell_relative(d.box, d.cells, x, c3);
    }
    return moved;
}

// (Bodies take the system d, this block's index bx among the gx blocks working
// on d, and stride over d's atoms.)

// Fold periodic coordinates into [0, L), bin into cells, count per cell.
__device__ __forceinline__ void cell_bin_atom(const Dev& d, int64_t i) {
    double4 x = d.x[i];
    double xs[3] = {x.x, x.y, x.z};
    for (int k = 0; k < 3; ++k)
        if (d.box.per[k]) xs[k] = __dsub_rn(xs[k], __dmul_rn(d.box.L[k], floor(__dmul_rn(xs[k], d.box.invL[k]))));
    x.x = xs[0];
    x.y = xs[1];
    x.z = xs[2];
    d.x[i] = x;
    d.xf[i] = make_float4((float)xs[0], (float)xs[1], (float)xs[2], 0.f);
    const int cx = cell_coord(d.box, d.cells, xs[0], 0);
    const int cy = cell_coord(d.box, d.cells, xs[1], 1);
    const int cz = cell_coord(d.box, d.cells, xs[2], 2);
    const int c = (cz * d.cells.nc[1] + cy) * d.cells.nc[0] + cx;
    d.cell_of[i] = c;
    const int c3 = cx | (cy << 10) | (cz << 20);
    d.cell3[i] = c3;
    d.xr[i] = cell_relative(d.box, d.cells, x, c3);
    atomicAdd(d.cell_count + c, 1);
}

// Exclusive scan of the cell counts (one block), zeroing counts and fill slots.
__device__ __forceinline__ void cell_scan_body(const Dev& d) {
    __shared__ int wsum[32];
    __shared__ int carry_s;
    const int tid = threadIdx.x, lane = tid & 31, warp = tid >> 5, nw = blockDim.x >> 5;
    if (tid == 0) {
        carry_s = 0;
        d.status[SW_MAXNB] = 0;
    }
    __syncthreads();
    const int nc = d.cells.ncell;
    for (int base = 0; base < nc; base += blockDim.x) {
        const int k = base + tid;
        const int v = k < nc ? d.cell_count[k] : 0;
        int incl = v;
        for (int o = 1; o < 32; o <<= 1) {
            int t = __shfl_up_sync(0xffffffffu, incl, o);
            if (lane >= o) incl += t;
        }
        if (lane == 31) wsum[warp] = incl;
        __syncthreads();
        if (warp == 0) {
            int w = lane < nw ? wsum[lane] : 0;
            for (int o = 1; o < 32; o <<= 1) {
                int t = __shfl_up_sync(0xffffffffu, w, o);
                if (lane >= o) w += t;
            }
            if (lane < nw) wsum[lane] = w;
        }
        __syncthreads();
        const int carry = carry_s;
        const int excl = carry + (warp > 0 ? wsum[warp - 1] : 0) + incl - v;
        if (k < nc) {
            d.cell_start[k] = excl;
            d.cell_fill[k] = 0;
            d.cell_count[k] = 0;
        }
        __syncthreads();
        if (tid == blockDim.x - 1) carry_s = excl + v;
        __syncthreads();
    }
    if (tid == 0) d.cell_start[nc] = carry_s;
}
__device__ __forceinline__ void cell_fill_body(const Dev& d, int bx, int gx) {
    for (int64_t i = bx * (int64_t)blockDim.x + threadIdx.x; i < d.n; i += (int64_t)gx * blockDim.x) {
        const int c = d.cell_of[i];
        const int slot = d.cell_start[c] + atomicAdd(d.cell_fill + c, 1);
        d.cell_atoms[slot] = (int)i;
    }
}
// One warp per atom: the 27-cell stencil is up to 18 contiguous runs of cells
// (9 rows (dz, dy), one or two runs along x each); lane r < 18 finds run r, a
// warp prefix sum numbers all candidates of all runs, and the lanes take 32
// consecutive candidates at a time across run boundaries (in run order, so the
// compacted row is the same as a run-by-run scan) with the next 32 loaded
// ahead.  Candidates with r2 < rlist2 are compacted into shared memory with a
// ballot; each lane then ranks its entries among the row (atom indices are
// distinct) and writes them to their sorted places.
__device__ __forceinline__ int pow2_cap(int cap) {
    int c = 32;
    while (c < cap) c <<= 1;
    return c;
}

constexpr int NB_RUNS = 18;

// The candidate test of the list build: the float screen (NbScreen), then the
// exact float64 test, r^2 formed as in the oracle, near the threshold.
__device__ __forceinline__ bool nb_accept(const Dev& d, const double4& xi, const float4& xif, const float4& xjf, int j) {
    float df[3] = {xjf.x - xif.x, xjf.y - xif.y, xjf.z - xif.z};
#pragma unroll
    for (int k = 0; k < 3; ++k)
        if (d.box.per[k]) df[k] -= d.nbs.L[k] * rintf(df[k] * d.nbs.iL[k]);
    const float r2f = df[0] * df[0] + df[1] * df[1] + df[2] * df[2];
    if (r2f < d.nbs.lo2 && !d.exact_lists) return true;
    if (r2f <= d.nbs.hi2 || d.exact_lists) {
        double dd[3];
        delta_rn(d.box, xi, d.x[j], dd);
        return norm2_rn(dd) < d.rlist2;
    }
    return false;
}

// The runs of the 27-cell stencil of cell (cx, cy, cz): lane r < NB_RUNS gets
// run r's first cell_atoms index t0 and length len (0 for an absent run):
// rows (dz, dy) of three cells along x, one or two runs each.
__device__ __forceinline__ void nb_run(const Dev& d, int cx, int cy, int cz, int lane, int& t0, int& len) {
    const int ncx = d.cells.nc[0], ncy = d.cells.nc[1], ncz = d.cells.nc[2];
    t0 = 0;
    len = 0;
    if (lane >= NB_RUNS) return;
    const int rr = lane >> 1, run = lane & 1;
    int qz = cz + rr / 3 - 1, qy = cy + rr % 3 - 1;
    bool in = true;
    if (d.box.per[2]) qz = (qz + ncz) % ncz;
    else in = qz >= 0 && qz < ncz;
    if (d.box.per[1]) qy = (qy + ncy) % ncy;
    else in = in && qy >= 0 && qy < ncy;
    // runs of cells along x: [a0, b0] and optionally [a1, b1]
    int a0, b0, a1 = 1, b1 = 0;
    if (d.box.per[0]) {
        if (cx == 0) { a0 = 0; b0 = 1; a1 = ncx - 1; b1 = ncx - 1; }
        else if (cx == ncx - 1) { a0 = ncx - 2; b0 = ncx - 1; a1 = 0; b1 = 0; }
        else { a0 = cx - 1; b0 = cx + 1; }
    } else {
        a0 = cx > 0 ? cx - 1 : 0;
        b0 = cx < ncx - 1 ? cx + 1 : ncx - 1;
    }
    const int ra = run == 0 ? a0 : a1, rb = run == 0 ? b0 : b1;
    if (in && ra <= rb) {
        const int row = (qz * ncy + qy) * ncx;
        t0 = d.cell_start[row + ra];
        len = d.cell_start[row + rb + 1] - t0;
    }
}

// The longest row a warp wrote, once at its end rather than once a row: reductions to
// one address run at some 3 ns each on this part, 60 us for 20,000 rows.
__device__ __forceinline__ void nb_report_max(const Dev& d, int most, int lane) {
    if (lane == 0 && most > 0) atomicMax(d.status + SW_MAXNB, most);
}

// The row of atom i from its cnt accepted candidates in buf (this warp's
// capp2 ints): capacity check, then each lane ranks its entries among the row
// (atom indices are distinct) and stores them at their sorted places.
__device__ __forceinline__ void nb_write_row(const Dev& d, int64_t i, const double4& xi, int cnt, int* buf, int lane) {
    const int cap = d.cap;
    if (lane == 0 && cnt > cap) set_status(d.status, ST_NBR_OVERFLOW);
    const int mlen = cnt < cap ? cnt : cap;
    // pad to whole 4-vectors with INT_MAX (ranks unaffected): m4 <= capp2
    const int m4 = (mlen + 3) & ~3;
    if (mlen + lane < m4) buf[mlen + lane] = INT_MAX;
    __syncwarp();
    int* row = d.nbr + i * (int64_t)cap;
    const int4* b4 = reinterpret_cast<const int4*>(buf);
    for (int p = lane; p < mlen; p += 32) {
        const int v = buf[p];
        int rank = 0;
        for (int q = 0; q < (m4 >> 2); ++q) {
            const int4 w = b4[q];
            rank += (w.x < v) + (w.y < v) + (w.z < v) + (w.w < v);
        }
        row[rank] = v;
    }
    if (lane == 0) {
        d.nnb[i] = mlen;
        d.xb[i] = xi;
    }
    __syncwarp();
}

template <int NBW>
__device__ __forceinline__ void neigh_build_body(const Dev& d, int bx, int gx, int capp2, int* sbuf) {
    __shared__ int s_runx[NBW][NB_RUNS];   // cell_atoms index of a run's first candidate, less its number
    __shared__ int s_runi[NBW][NB_RUNS];   // candidates in runs 0..r
    const int lane = threadIdx.x & 31, warp = threadIdx.x >> 5;
    int* buf = sbuf + warp * capp2;
    int* runx = s_runx[warp];
    int* runi = s_runi[warp];
    const unsigned lt = (1u << lane) - 1u;
    const int ncx = d.cells.nc[0], ncy = d.cells.nc[1];
    int most = 0;
    for (int64_t i = (int64_t)bx * NBW + warp; i < d.n; i += (int64_t)gx * NBW) {
        const double4 xi = d.x[i];
        const float4 xif = d.xf[i];
        const int c = d.cell_of[i];
        const int cx = c % ncx, cy = (c / ncx) % ncy, cz = c / (ncx * ncy);
        int len, t0;
        nb_run(d, cx, cy, cz, lane, t0, len);
        int inc = len;
#pragma unroll
        for (int o = 1; o < 32; o <<= 1) {
            const int v = __shfl_up_sync(0xffffffffu, inc, o);
            if (lane >= o) inc += v;
        }
        const int total = __shfl_sync(0xffffffffu, inc, 31);
        if (lane < NB_RUNS) {
            runi[lane] = inc;
            runx[lane] = t0 - (inc - len);
        }
        __syncwarp();
        // the atom one pass ahead is loaded before this pass is tested (r: run of the
        // furthest candidate loaded)
        int r = 0;
        int jn = -1;
        if (lane < total) {
            while (lane >= runi[r]) ++r;
            jn = d.cell_atoms[runx[r] + lane];
        }
        int cnt = 0;
        for (int u = lane; u - lane < total; u += 32) {
            const int j = jn;
            if (u + 32 < total) {
                while (u + 32 >= runi[r]) ++r;
                jn = d.cell_atoms[runx[r] + u + 32];
            }
            bool ok = false;
            if (u < total && j != (int)i) ok = nb_accept(d, xi, xif, d.xf[j], j);
            const unsigned m = __ballot_sync(0xffffffffu, ok);
            if (ok) {
                const int p = cnt + __popc(m & lt);
                if (p < capp2) buf[p] = j;
            }
            cnt += __popc(m);
        }
        nb_write_row(d, i, xi, cnt, buf, lane);
        most = max(most, cnt);
    }
    nb_report_max(d, most, lane);
}

// The list build of a single context with neighbour-cell tiles staged in shared
// memory: a team of NB_TEAM warps takes a cell at a time, copies the candidates of its
// 27-cell stencil (float position and atom index, in run order) into shared memory
// once, and its warps take the cell's atoms, a warp per atom, testing 32
// staged candidates at a time; the candidates cross L2 once per cell instead
// of once per atom.  A CTA of 16 warps is four teams that do not wait for each
// other: a cell holds some 8 atoms in silicon and 17 in iron, so 16 warps on one cell
// left half of them idle (evaluations that rebuild, front, us, 16 warps a cell / 8 / 4 /
// 2: 20,383 silicon atoms 92 / 82 / 81 / 95, 499,199 of them 1247 / 899 / 802 / 1090, 50,459
// iron atoms 234 / 214 / 223 / 294, 198,903 of them 691 / 628 / 613 / 840, 998,559 of them
// 3606 / 3046 / 2935 / 4087).  The staged positions are taken relative to the cell's centre,
// each as the periodic image next to it, so that the test of a pair is a
// difference and three products (a periodic dimension has at least four cells
// here, nb_tiled_ok, each at least as wide as the list radius: the stencil lies
// well inside half a box of the centre, so a pair closer than the radius is found
// at those images and any other pair only reads as farther away): the minimum image
// per pair and component was half the instructions of this issue-bound kernel.
// The float screen only decides away from the threshold, so the rows are those of
// the warp-per-atom build (neigh_build_body).  A stencil with more than NB_TILE
// candidates (a dense spot) is tested from global memory instead.
constexpr int NB_TILE = 1024;
constexpr int NB_TEAM = 4;

inline bool nb_tiled_ok(const Dev& d) {
    for (int k = 0; k < 3; ++k)
        if (d.box.per[k] && d.cells.nc[k] < 4) return false;
    return true;
}

inline size_t nb_tiled_smem(int capp2, int warps) {
    return (size_t)NB_TILE * (warps / NB_TEAM) * sizeof(float4) + (size_t)warps * capp2 * sizeof(int);
}

// barrier of one team (the CTA's barrier is number 0)
__device__ __forceinline__ void nb_team_sync(int team) {
    asm volatile("bar.sync %0, %1;" ::"r"(team + 1), "n"(NB_TEAM * 32) : "memory");
}

template <int NBW>
__device__ __forceinline__ void neigh_build_tiled_body(const Dev& d, int bx, int gx, int capp2, unsigned char* nb_smem) {
    constexpr int NT = NBW / NB_TEAM;
    const int lane = threadIdx.x & 31, warp = threadIdx.x >> 5, team = warp / NB_TEAM, tw = warp % NB_TEAM;
    float4* tile = reinterpret_cast<float4*>(nb_smem) + team * NB_TILE;   // position, atom index in w
    int* buf = reinterpret_cast<int*>(reinterpret_cast<float4*>(nb_smem) + NT * NB_TILE) + warp * capp2;
    __shared__ int s_runx[NT][NB_RUNS], s_runi[NT][NB_RUNS];
    int* runx = s_runx[team];
    int* runi = s_runi[team];
    const unsigned lt = (1u << lane) - 1u;
    const int ncx = d.cells.nc[0], ncy = d.cells.nc[1];
    const int ncell = d.cells.ncell;
    int most = 0;
    for (int c = bx * NT + team; c < ncell; c += gx * NT) {
        const int a0 = d.cell_start[c], a1 = d.cell_start[c + 1];
        if (a0 == a1) continue;   // the same for the whole team
        const int cx = c % ncx, cy = (c / ncx) % ncy, cz = c / (ncx * ncy);
        if (tw == 0) {
            int t0, len;
            nb_run(d, cx, cy, cz, lane, t0, len);
            int inc = len;
#pragma unroll
            for (int o = 1; o < 32; o <<= 1) {
                const int v = __shfl_up_sync(0xffffffffu, inc, o);
                if (lane >= o) inc += v;
            }
            if (lane < NB_RUNS) {
                runi[lane] = inc;
                runx[lane] = t0 - (inc - len);
            }
        }
        // the cell's centre, and a position as its periodic image next to it
        const float ctr[3] = {d.nbs.lo[0] + (cx + 0.5f) * d.cells.hf[0], d.nbs.lo[1] + (cy + 0.5f) * d.cells.hf[1],
                              d.nbs.lo[2] + (cz + 0.5f) * d.cells.hf[2]};
        auto relative = [&](const float4& x) {
            float v[3] = {x.x - ctr[0], x.y - ctr[1], x.z - ctr[2]};
#pragma unroll
            for (int k = 0; k < 3; ++k)
                if (d.box.per[k]) v[k] -= d.nbs.L[k] * rintf(v[k] * d.nbs.iL[k]);
            return make_float4(v[0], v[1], v[2], 0.f);
        };
        nb_team_sync(team);
        const int total = runi[NB_RUNS - 1];
        const bool staged = total <= NB_TILE;
        if (staged) {
            int r = 0;
            for (int t = tw * 32 + lane; t < total; t += NB_TEAM * 32) {
                while (t >= runi[r]) ++r;
                const int j = d.cell_atoms[runx[r] + t];
                float4 v = relative(d.xf[j]);
                v.w = __int_as_float(j);
                tile[t] = v;
            }
        }
        nb_team_sync(team);
        for (int a = a0 + tw; a < a1; a += NB_TEAM) {
            const int i = d.cell_atoms[a];
            const double4 xi = d.x[i];
            const float4 xif = d.xf[i];
            const float4 ri = relative(xif);
            int cnt = 0;
            int r = 0;
            for (int u = lane; u - lane < total; u += 32) {
                bool ok = false;
                int j = -1;
                if (u < total) {
                    if (staged) {
                        const float4 rj = tile[u];
                        j = __float_as_int(rj.w);
                        const float dx = rj.x - ri.x, dy = rj.y - ri.y, dz = rj.z - ri.z;
                        const float r2f = dx * dx + dy * dy + dz * dz;
                        ok = r2f < d.nbs.lo2;
                        if (d.exact_lists || (!ok && r2f <= d.nbs.hi2)) {
                            double dd[3];
                            delta_rn(d.box, xi, d.x[j], dd);
                            ok = norm2_rn(dd) < d.rlist2;
                        }
                        ok = ok && j != i;
                    } else {
                        while (u >= runi[r]) ++r;
                        j = d.cell_atoms[runx[r] + u];
                        if (j != i) ok = nb_accept(d, xi, xif, d.xf[j], j);
                    }
                }
                const unsigned m = __ballot_sync(0xffffffffu, ok);
                if (ok) {
                    const int p = cnt + __popc(m & lt);
                    if (p < capp2) buf[p] = j;
                }
                cnt += __popc(m);
            }
            nb_write_row(d, i, xi, cnt, buf, lane);
            most = max(most, cnt);
        }
        nb_team_sync(team);   // the tile and the runs are rewritten for the next cell
    }
    nb_report_max(d, most, lane);
}

// rev[i][s] = position of i in the row of j = nbr[i][s] (binary search in the
// sorted row).  A warp per atom, lanes over its row's slots.
__device__ __forceinline__ void neigh_rev_body(const Dev& d, int bx, int gx) {
    const int lane = threadIdx.x & 31, wpb = (int)(blockDim.x >> 5);
    const int cap = d.cap;
    for (int64_t i = (int64_t)bx * wpb + (threadIdx.x >> 5); i < d.n; i += (int64_t)gx * wpb) {
        const int m = d.nnb[i];
        const int* ri = d.nbr + i * cap;
        for (int s = lane; s < m; s += 32) {
            const int j = ri[s];
            const int* row = d.nbr + (int64_t)j * cap;
            int lo = 0, hi = d.nnb[j] - 1, pos = -1;
            while (lo <= hi) {
                const int mid = (lo + hi) >> 1;
                const int v = row[mid];
                if (v == (int)i) {
                    pos = mid;
                    break;
                }
                if (v < (int)i) lo = mid + 1;
                else hi = mid - 1;
            }
            if (pos < 0) {
                set_status(d.status, ST_REV_MISSING);
                pos = 0;
            }
            d.rev[i * cap + s] = pos;
        }
    }
}

}  // namespace mixd
