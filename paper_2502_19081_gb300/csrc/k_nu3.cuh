// The float nu = 3 pass of one l-triple for one atom (a warp), in three phases:
//   U:   U[m3][q1][q2] = sum_q3 W[q1 q2][q3] A3[m3][q3]      (dense, rolled over m3)
//   mid: Z[m3][q1][q2] = sum_m2 B[m3][m2] A2[m2][q2],  B[m3][m2] = sum_m1 G A1[m1][q1],
//        omega1[m1][q1] += G sum_q2 A2[m2][q2] U[m3][q1][q2],
//        omega2[m2][q2] += sum_(q1 m3) B[m3][m2] U[m3][q1][q2]   (distinct l's only)
//        with the Gaunt pattern of the triple known at compile time;
//   W:   omega3[m3][q3] += sum_(q1 q2) W[q1 q2][q3] Z[m3][q1][q2],  E += sum A3 (W^T Z).
// A lane owns one unit (q1, QB consecutive q2) in all three, and U and Z pass
// between the phases through the unit's own places of a shared-memory row
// buffer (Z overwrites U), so no phase holds another's registers.
//
// Why: issue slots bound this kernel, not the FMA pipe.  With the Gaunt entries
// read from a table an entry cost some 35 instructions (decode, address
// arithmetic, a read-modify-write of the omega1 partial in shared memory, loop
// control) for the 7 multiply-adds it is there for.  Which real Gaunt
// coefficients are non-zero follows from the signs and sizes of the m's alone,
// so the phase "mid" is unrolled over (m2, m3): A1 and the omega1 partials sit
// in registers, an (m2, m3) pair takes its one or two coefficients as
// constant-bank operands, and its value B serves Z and omega2.  The dense phases
// choose their own lanes: U a W row per lane, W a split of (q1 q2) per lane pair.
// Splitting the phases also brings the registers from 160 to 128 a thread, so
// 16 warps share an SM instead of 12.
// Measured (n = 12, lmax = 5, 19,284 atoms evaluated, float): 1.96 -> 1.06 ms a
// launch, 1.36 -> 0.66 G instructions; n = 10, lmax = 4, 1,394 atoms: 112 -> 80 us
// (a warp an atom and nine atoms an SM: one atom's latency); with the bf16
// readout, n = 12, 256,000-atom cylinder: 2.71 -> 1.95 ms with the cheap kernel
// inside.
#pragma once

#include <utility>

#include "mix_dev.cuh"
#include "tc.cuh"

namespace mixd {

// ---------------------------------------------------------------------------
// The compile-time pattern: m's run from -l to l (m < 0: the sine functions).
// G(l1 m1, l2 m2, l3 m3) is zero unless the number of sines is even and
// |m1| = |m2| + |m3| or ||m2| - |m3||; for given m2, m3 that leaves at most two m1.

constexpr int gp_abs(int a) { return a < 0 ? -a : a; }

// the k-th (k = 0, 1) m1 of the pair (m2, m3), or l1 + 1 when there is none;
// the smaller |m1| first
__host__ __device__ constexpr int gp_m1(int l1, int m2, int m3, int k) {
    const bool neg = (m2 < 0) != (m3 < 0);
    const int a = m2 < 0 ? -m2 : m2, b = m3 < 0 ? -m3 : m3;
    const int lo = a > b ? a - b : b - a, hi = a + b;
    int found = 0;
    for (int t = 0; t < 2; ++t) {
        const int v = t == 0 ? lo : hi;
        if (t == 1 && hi == lo) continue;
        if (v > l1 || (neg && v == 0)) continue;
        if (found == k) return neg ? -v : v;
        ++found;
    }
    return l1 + 1;
}
__host__ __device__ constexpr int gp_count(int l1, int m2, int m3) {
    return (gp_m1(l1, m2, m3, 0) <= l1 ? 1 : 0) + (gp_m1(l1, m2, m3, 1) <= l1 ? 1 : 0);
}

// the l-triples l1 >= l2 >= l3 (even sum, l1 <= l2 + l3) up to MIX_MAX_LMAX, in
// the order l3, l2, l1 ascending
struct TriL {
    int l1, l2, l3;
};
__host__ __device__ constexpr TriL tri_l(int id) {
    int k = 0;
    for (int l3 = 0; l3 <= MIX_MAX_LMAX; ++l3)
        for (int l2 = l3; l2 <= MIX_MAX_LMAX; ++l2)
            for (int l1 = l2; l1 <= MIX_MAX_LMAX; ++l1) {
                if (((l1 + l2 + l3) & 1) || l1 > l2 + l3) continue;
                if (k == id) return TriL{l1, l2, l3};
                ++k;
            }
    return TriL{-1, -1, -1};
}
constexpr int TRI_COUNT = 30;
static_assert(tri_l(TRI_COUNT - 1).l1 == MIX_MAX_LMAX && tri_l(TRI_COUNT).l1 < 0, "number of l-triples");

__host__ __device__ constexpr int tri_values(int l1, int l2, int l3) {
    int n = 0;
    for (int m2 = -l2; m2 <= l2; ++m2)
        for (int m3 = -l3; m3 <= l3; ++m3) n += gp_count(l1, m2, m3);
    return n;
}
// first coefficient of triple id in the table (ordered by triple, m2, m3, k)
__host__ __device__ constexpr int tri_first(int id) {
    int n = 0;
    for (int t = 0; t < id; ++t) {
        const TriL l = tri_l(t);
        n += tri_values(l.l1, l.l2, l.l3);
    }
    return n;
}
constexpr int GP_COUNT = 1938;
static_assert(tri_first(TRI_COUNT) == GP_COUNT, "number of Gaunt coefficients in the pattern");

// where the coefficients of every pair (m2, m3) of a triple start
template <int L1, int L2, int L3>
struct TriTab {
    int at[2 * L2 + 1][2 * L3 + 1] = {};
    __host__ __device__ constexpr explicit TriTab(int first) {
        for (int m2 = -L2; m2 <= L2; ++m2)
            for (int m3 = -L3; m3 <= L3; ++m3) {
                at[m2 + L2][m3 + L3] = first;
                first += gp_count(L1, m2, m3);
            }
    }
};

template <int ID>
struct TriC {
    static constexpr TriL l = tri_l(ID);
    static constexpr TriTab<l.l1, l.l2, l.l3> tab{tri_first(ID)};
};

// the coefficients: a copy in the constant memory of each module that holds the
// float expensive kernels, read as immediate-offset operands
static __constant__ float c_gp[GP_COUNT];

// this module's copy of the table (host side)
static inline cudaError_t gaunt_upload_module(const float* g, int n) {
    if (n != GP_COUNT) return cudaErrorInvalidValue;
    return cudaMemcpyToSymbol(c_gp, g, (size_t)n * sizeof(float));
}

template <class F, int... I>
__device__ __forceinline__ void sfor_impl(F&& f, std::integer_sequence<int, I...>) {
    (f(std::integral_constant<int, I>{}), ...);
}
// f(0), f(1), ..., f(N - 1) with compile-time arguments
template <int N, class F>
__device__ __forceinline__ void sfor(F&& f) {
    sfor_impl(f, std::make_integer_sequence<int, N>{});
}

// ---------------------------------------------------------------------------

// Reduce-scatter of C <= 16 per-lane values over the warp.  At lane bit MASK
// (16, 8, 4, 2, 1 in turn, down to END) the lanes with the bit set keep the upper half of
// their block (padded with a zero when the count is odd) and send the lower
// half to their partner, the others the reverse, and each adds what it
// receives, so the count halves at every bit; once one value is left the
// remaining bits sum it (both partners add the same two numbers).  The
// additions are in a fixed order.  rs_entry gives the entry a lane ends with.
template <typename T, int C, int MASK, int END = 1>
__device__ __forceinline__ T warp_rs(T* v, int lane) {
    if constexpr (MASK < END) {
        return v[0];
    } else if constexpr (C == 1) {
        v[0] += __shfl_xor_sync(0xffffffffu, v[0], MASK);
        return warp_rs<T, 1, MASK / 2, END>(v, lane);
    } else {
        constexpr int H = (C + 1) / 2;
        const bool up = (lane & MASK) != 0;
#pragma unroll
        for (int i = 0; i < H; ++i) {
            const T hi = i + H < C ? v[i + H] : T(0);
            const T send = up ? v[i] : hi;
            const T keep = up ? hi : v[i];
            v[i] = keep + __shfl_xor_sync(0xffffffffu, send, MASK);
        }
        return warp_rs<T, H, MASK / 2, END>(v, lane);
    }
}

// The entry of warp_rs<T, C, 16> a lane holds (idx), and whether the lane is
// the one of its group that writes it (a real entry, the lowest lane of the
// lanes that hold the same sum).
template <int C, int MASK, int END = 1>
__device__ __forceinline__ void rs_entry(int lane, int& idx, int& real, bool& writer) {
    if constexpr (MASK < END) {
        writer = real >= 1;
    } else if constexpr (C == 1) {
        writer = real >= 1 && (lane & (2 * MASK - 1) & ~(END - 1)) == 0;
    } else {
        constexpr int H = (C + 1) / 2;
        if (lane & MASK) {
            idx += H;
            real = real > H ? real - H : 0;
        } else {
            real = real < H ? real : H;
        }
        rs_entry<H, MASK / 2, END>(lane, idx, real, writer);
    }
}

// The q2 block of a lane unit for n radial functions in rows padded to np: a
// warp covers the units in one pass (n np / qb <= 32) with as few idle lanes
// as aligned pairs allow: n <= 4: 2, n <= 8: 2, n <= 10: 4, n <= 12: 6, n <= 16: 8.
__host__ __device__ constexpr int nu3_qb(int n) { return n <= 8 ? 2 : (n <= 10 ? 4 : (n <= 12 ? 6 : 8)); }

// q3 values the dense phases run over (n rounded up to a pair; the row padding
// beyond them is skipped): 10 of the 12 for n <= 10
template <int NP, int QB>
__host__ __device__ constexpr int nu3_nq() {
    return NP == 12 && QB == 4 ? 10 : NP;
}

// rows of the U / Z buffer for a potential of lmax L: at most 2 l3 + 1 (U, Z),
// and for three distinct l's 2 l2 + 1 <= 2 L - 1 (the omega2 partials)
__host__ __device__ constexpr int nu3_rows(int L) {
    int r = 1;
    for (int t = 0; t < TRI_COUNT; ++t) {
        const TriL l = tri_l(t);
        if (l.l1 > L) continue;
        const int v = (l.l1 > l.l2 && l.l2 > l.l3) ? 2 * l.l2 + 1 : 2 * l.l3 + 1;
        r = v > r ? v : r;
    }
    return r;
}

// a lane's unit
struct Nu3Unit {
    int q1, q2;
    bool uv;
};
template <int NP, int QB>
__device__ __forceinline__ Nu3Unit nu3_unit(int n, int lane) {
    constexpr int nqb = NP / QB;
    Nu3Unit u;
    u.uv = lane < n * nqb;
    const int uu = u.uv ? lane : 0;
    u.q1 = uu / nqb;
    u.q2 = (uu - u.q1 * nqb) * QB;
    return u;
}

// QB consecutive floats (QB even, 8-byte aligned; QB a multiple of 4: 16-byte
// aligned) as pairs
template <int QB>
__device__ __forceinline__ void ld_pairs(const float* p, float2* out) {
    if constexpr (QB % 4 == 0) {
#pragma unroll
        for (int k = 0; k < QB / 4; ++k) {
            const float4 v = reinterpret_cast<const float4*>(p)[k];
            out[2 * k] = make_float2(v.x, v.y);
            out[2 * k + 1] = make_float2(v.z, v.w);
        }
    } else {
#pragma unroll
        for (int k = 0; k < QB / 2; ++k) out[k] = reinterpret_cast<const float2*>(p)[k];
    }
}
template <int QB>
__device__ __forceinline__ void st_pairs(float* p, const float2* v) {
    if constexpr (QB % 4 == 0) {
#pragma unroll
        for (int k = 0; k < QB / 4; ++k)
            reinterpret_cast<float4*>(p)[k] = make_float4(v[2 * k].x, v[2 * k].y, v[2 * k + 1].x, v[2 * k + 1].y);
    } else {
#pragma unroll
        for (int k = 0; k < QB / 2; ++k) reinterpret_cast<float2*>(p)[k] = v[k];
    }
}

// NQ values of a 16-byte aligned row as pairs
template <int NQ>
__device__ __forceinline__ void ld_row(const float* p, float2* out) {
#pragma unroll
    for (int k = 0; k < NQ / 4; ++k) {
        const float4 v = reinterpret_cast<const float4*>(p)[k];
        out[2 * k] = make_float2(v.x, v.y);
        out[2 * k + 1] = make_float2(v.z, v.w);
    }
    if constexpr (NQ % 4 != 0) out[NQ / 2 - 1] = reinterpret_cast<const float2*>(p)[NQ / 2 - 1];
}

// Rows of the flattened index k = q1 NP + q2 (n NP of them; the W rows of the
// padding q2 >= n are zero) a lane takes in phase U (a row per lane) and k's a
// lane takes in phase W (16 splits of k, a lane pair each), by class
template <int NP, int QB>
__host__ __device__ constexpr int nu3_kmax() {
    return (NP == 12 && QB == 4 ? 10 : NP) * NP;
}
// the least n NP of the class: k's below it need no test
template <int NP, int QB>
__host__ __device__ constexpr int nu3_kmin() {
    return (NP == 4 ? 1 : NP == 8 ? 5 : NP == 16 ? 13 : (QB == 4 ? 9 : 11)) * NP;
}
template <int NP, int QB>
__host__ __device__ constexpr int nu3_ku() {
    return (nu3_kmax<NP, QB>() + 31) / 32;
}
template <int NP, int QB>
__host__ __device__ constexpr int nu3_kw() {
    return (nu3_kmax<NP, QB>() + 15) / 16;
}

// Phase U: rows m3 = 0 .. d3 - 1 of the buffer.  Lane l takes the rows
// k = l, l + 32, ..: consecutive lanes read consecutive 4 NP-byte rows of W, which
// spreads a 16-byte read over all banks, and all 32 lanes work.
template <int NP, int QB>
__device__ __forceinline__ void nu3_dense_u(const float* W, const float* A3, int n, int d3, int lane, float* uz) {
    constexpr int NQ = nu3_nq<NP, QB>(), NH = NQ / 2, KU = nu3_ku<NP, QB>(), KMIN = nu3_kmin<NP, QB>();
    const int kn = n * NP;
    float2 w[KU][NH];
#pragma unroll
    for (int i = 0; i < KU; ++i) {
        const int k = lane + 32 * i;
        ld_row<NQ>(W + (k < kn ? k : 0) * NP, w[i]);
    }
    float* p = uz + lane;
    // two rows m3 at a time (independent chains), then the odd one
    auto rows = [&](auto rc) {
        constexpr int R = rc.value;
        float2 a[R][NH];
#pragma unroll
        for (int r = 0; r < R; ++r) ld_row<NQ>(A3 + r * NP, a[r]);
#pragma unroll
        for (int i = 0; i < KU; ++i) {
#pragma unroll
            for (int r = 0; r < R; ++r) {
                float2 s = make_float2(0.f, 0.f);
#pragma unroll
                for (int j = 0; j < NH; ++j) s = __ffma2_rn(w[i][j], a[r][j], s);
                if (32 * i + 31 < KMIN || lane + 32 * i < kn) p[r * kn + 32 * i] = s.x + s.y;
            }
        }
    };
    int m3 = 0;
    for (; m3 + 2 <= d3; m3 += 2, A3 += 2 * NP, p += 2 * kn) rows(std::integral_constant<int, 2>{});
    if (m3 < d3) rows(std::integral_constant<int, 1>{});
    __syncwarp();
}

// Phase W: omega3 and the energy from the rows Z of the buffer.  Lane pair g
// takes k = g, g + 16, .., lane t of the pair one half of the q3's, so that an
// m3 row ends in a reduction of NP / 2 values over 16 pairs (7 shuffles for NP =
// 12; with a lane per unit and all q3's it took 13) and no lane is idle.  Two rows
// are reduced together: the four dependent shuffle rounds are the row's critical
// path where few warps share an SM.
template <int NP, int QB>
__device__ __forceinline__ void nu3_dense_w(const float* W, const float* A3, int n, int d3, const float* uz, float* o3,
                                            float mult3, int lane, float& ep) {
    constexpr int HQ = NP / 2, HP = HQ / 2, KW = nu3_kw<NP, QB>(), KMIN = nu3_kmin<NP, QB>();
    const int kn = n * NP, g = lane >> 1, t0 = (lane & 1) * HQ;
    float2 w[KW][HP];
#pragma unroll
    for (int i = 0; i < KW; ++i) {
        const int k = g + 16 * i;
        const float2* r = reinterpret_cast<const float2*>(W + (k < kn ? k : 0) * NP + t0);
#pragma unroll
        for (int j = 0; j < HP; ++j) w[i][j] = k < kn ? r[j] : make_float2(0.f, 0.f);
    }
    const float* p = uz + g;
    auto rows = [&](auto rc, int m3) {
        constexpr int R = rc.value;
        float2 s[R][HP];
#pragma unroll
        for (int r = 0; r < R; ++r)
#pragma unroll
            for (int j = 0; j < HP; ++j) s[r][j] = make_float2(0.f, 0.f);
#pragma unroll
        for (int i = 0; i < KW; ++i) {
#pragma unroll
            for (int r = 0; r < R; ++r) {
                const float z = 16 * i + 15 < KMIN || g + 16 * i < kn ? p[r * kn + 16 * i] : 0.f;
#pragma unroll
                for (int j = 0; j < HP; ++j) s[r][j] = __ffma2_rn(w[i][j], make_float2(z, z), s[r][j]);
            }
        }
        float pv[R * HQ];
#pragma unroll
        for (int r = 0; r < R; ++r)
#pragma unroll
            for (int j = 0; j < HP; ++j) {
                pv[r * HQ + 2 * j] = s[r][j].x;
                pv[r * HQ + 2 * j + 1] = s[r][j].y;
            }
        int o = 0, real = R * HQ;   // the entry (row, q3) this lane receives
        bool wr = false;
        rs_entry<R * HQ, 16, 2>(lane, o, real, wr);
        const float s3 = warp_rs<float, R * HQ, 16, 2>(pv, lane);
        const int r = o >= HQ ? 1 : 0, q = o - r * HQ + t0;
        if (wr && q < n) {
            o3[(m3 + r) * NP + q] += mult3 * s3;
            ep += A3[(m3 + r) * NP + q] * s3;
        }
    };
    int m3 = 0;
    for (; m3 + 2 <= d3; m3 += 2, p += 2 * kn) rows(std::integral_constant<int, 2>{}, m3);
    if (m3 < d3) rows(std::integral_constant<int, 1>{}, m3);
    __syncwarp();
}

// Where Z goes for the tensor-core readout: this atom's rows of the MMA operand
// tile (row m3, column q1 n + q2, K-major layout of tc.cuh), rounded to bf16;
// TCM == 2 also the remainders.
struct Nu3Op {
    unsigned char* hi;
    unsigned char* lo;
    int sbo;
};

template <int QB, int TCM>
__device__ __forceinline__ void nu3_st_op(const Nu3Op& op, int m3, int n, const Nu3Unit& u, const float2* z) {
    if ((n & 1) == 0) {
        // even n: each pair of columns lies in one 4-byte word of a core-matrix row
#pragma unroll
        for (int k = 0; k < QB / 2; ++k) {
            if (u.q2 + 2 * k < n) {
                const int o = tc_off(m3, u.q1 * n + u.q2 + 2 * k, TC_LBO_A, op.sbo);
                const __nv_bfloat162 hi = __float22bfloat162_rn(z[k]);
                *reinterpret_cast<__nv_bfloat162*>(op.hi + o) = hi;
                if constexpr (TCM == 2) {
                    const float2 hf = __bfloat1622float2(hi);
                    *reinterpret_cast<__nv_bfloat162*>(op.lo + o) =
                        __float22bfloat162_rn(make_float2(z[k].x - hf.x, z[k].y - hf.y));
                }
            }
        }
    } else {
#pragma unroll
        for (int r = 0; r < QB; ++r) {
            if (u.q2 + r < n) {
                const float zr = (r & 1) ? z[r / 2].y : z[r / 2].x;
                const int o = tc_off(m3, u.q1 * n + u.q2 + r, TC_LBO_A, op.sbo);
                const __nv_bfloat16 hi = __float2bfloat16_rn(zr);
                *reinterpret_cast<__nv_bfloat16*>(op.hi + o) = hi;
                if constexpr (TCM == 2)
                    *reinterpret_cast<__nv_bfloat16*>(op.lo + o) = __float2bfloat16_rn(zr - __bfloat162float(hi));
            }
        }
    }
}

// omega2 of a triple of distinct l's: the buffer's rows m2 hold the units'
// partials, summed over q1 (in order) by a lane per (m2, pair of q2)
template <int NP>
__device__ __forceinline__ void nu3_omega2(const float* uz, float* o2, int n, int d2, int lane) {
    constexpr int NH = NP / 2;
    for (int o = lane; o < d2 * NH; o += 32) {
        const int m2 = o / NH, j = (o - m2 * NH) * 2;
        const float* p = uz + m2 * n * NP + j;
        float2 s = make_float2(0.f, 0.f);
#pragma unroll 4
        for (int q1 = 0; q1 < n; ++q1) {
            const float2 v = *reinterpret_cast<const float2*>(p + q1 * NP);
            s.x += v.x;
            s.y += v.y;
        }
        float2* r = reinterpret_cast<float2*>(o2 + m2 * NP + j);
        float2 t = *r;
        t.x += s.x;
        if (j + 1 < n) t.y += s.y;
        if (j < n) *r = t;
    }
}

// phase mid of triple ID.  m3 is taken in chunks so that U and Z of a chunk
// stay in registers (all of it for distinct l's, whose omega2 partials then
// overwrite the U rows).
template <int ID, int NP, int QB, int TCM>
__device__ __noinline__ void nu3_mid(const float* At, float* om, float* uz, int n, int lane, const Nu3Op op) {
    constexpr TriL T = tri_l(ID);
    constexpr int L1 = T.l1, L2 = T.l2, L3 = T.l3;
    constexpr int D1 = 2 * L1 + 1, D2 = 2 * L2 + 1, D3 = 2 * L3 + 1;
    constexpr int MODE = (L1 == L2 && L2 == L3) ? 3 : (L1 == L2 ? 1 : (L2 == L3 ? 2 : 0));
    constexpr int QH = QB / 2, nqb = NP / QB;
    constexpr int CM = QB <= 4 ? 9 : (QB == 6 ? (D1 >= 11 ? 3 : 5) : 4) * (MODE == 3 ? 2 : 1);
    constexpr int NC = MODE == 0 ? 1 : (D3 + CM - 1) / CM;   // chunks of m3
    constexpr int C = (D3 + NC - 1) / NC;
    const Nu3Unit u = nu3_unit<NP, QB>(n, lane);
    const float* A1 = At + L1 * L1 * NP + u.q1;
    const float* A2 = At + L2 * L2 * NP + u.q2;
    float* row = uz + u.q1 * NP + u.q2;
    const int rs = n * NP;   // row stride
    float a1[D1], p1[D1];
#pragma unroll
    for (int m = 0; m < D1; ++m) {
        a1[m] = A1[m * NP];
        p1[m] = 0.f;
    }
    sfor<NC>([&](auto ci) {
        constexpr int m30 = ci.value * C, CN = m30 + C <= D3 ? C : D3 - m30;
        [[maybe_unused]] float2 uu[CN][QH];
        float2 z[CN][QH];
#pragma unroll
        for (int c = 0; c < CN; ++c) {
            if constexpr (MODE != 3) ld_pairs<QB>(row + (m30 + c) * rs, uu[c]);
#pragma unroll
            for (int k = 0; k < QH; ++k) z[c][k] = make_float2(0.f, 0.f);
        }
        sfor<D2>([&](auto m2i) {
            constexpr int m2 = m2i.value;
            float2 a2[QH];
            [[maybe_unused]] float2 t[QH];
            ld_pairs<QB>(A2 + m2 * NP, a2);
#pragma unroll
            for (int k = 0; k < QH; ++k) t[k] = make_float2(0.f, 0.f);
            sfor<CN>([&](auto cc) {
                constexpr int c = cc.value, m3 = m30 + c;
                constexpr int cnt = gp_count(L1, m2 - L2, m3 - L3);
                if constexpr (cnt > 0) {
                    constexpr int at = TriC<ID>::tab.at[m2][m3];
                    constexpr int ma = gp_m1(L1, m2 - L2, m3 - L3, 0) + L1;
                    constexpr int mb = cnt > 1 ? gp_m1(L1, m2 - L2, m3 - L3, 1) + L1 : ma;
                    float b = c_gp[at] * a1[ma];
                    if constexpr (cnt > 1) b = fmaf(c_gp[at + 1], a1[mb], b);
                    const float2 b2 = make_float2(b, b);
#pragma unroll
                    for (int k = 0; k < QH; ++k) z[c][k] = __ffma2_rn(b2, a2[k], z[c][k]);
                    if constexpr (MODE == 0) {
#pragma unroll
                        for (int k = 0; k < QH; ++k) t[k] = __ffma2_rn(b2, uu[c][k], t[k]);
                    }
                    if constexpr (MODE != 3) {
                        float2 dd = make_float2(0.f, 0.f);
#pragma unroll
                        for (int k = 0; k < QH; ++k) dd = __ffma2_rn(a2[k], uu[c][k], dd);
                        const float s = dd.x + dd.y;
                        p1[ma] = fmaf(c_gp[at], s, p1[ma]);
                        if constexpr (cnt > 1) p1[mb] = fmaf(c_gp[at + 1], s, p1[mb]);
                    }
                }
            });
            if constexpr (MODE == 0) {
                if (u.uv) st_pairs<QB>(row + m2 * rs, t);
            }
        });
        if constexpr (TCM == 0) {
            if constexpr (MODE == 0) {
                __syncwarp();
                nu3_omega2<NP>(uz, om + L2 * L2 * NP, n, D2, lane);
                __syncwarp();
            }
            if (u.uv) {
#pragma unroll
                for (int c = 0; c < CN; ++c) st_pairs<QB>(row + (m30 + c) * rs, z[c]);
            }
        } else if (u.uv) {
#pragma unroll
            for (int c = 0; c < CN; ++c) nu3_st_op<QB, TCM>(op, m30 + c, n, u, z[c]);
        }
    });
    // omega1 (equal to omega3 when all three l's coincide): the partials of the
    // units of one q1, which are neighbouring lanes, summed in order
    if constexpr (MODE != 3) {
        float* o1 = om + L1 * L1 * NP + u.q1;
        const bool wr = u.uv && u.q2 == 0;
#pragma unroll
        for (int m = 0; m < D1; ++m) {
            float s = p1[m];
#pragma unroll
            for (int k = 1; k < nqb; ++k) s += __shfl_down_sync(0xffffffffu, p1[m], k);
            if (wr) o1[m * NP] += MODE == 1 ? 2.f * s : s;
        }
    }
    __syncwarp();
}

// run-time triple -> nu3_mid (triples beyond the kernel's lmax are not compiled in)
template <int L, int NP, int QB, int TCM>
__device__ __forceinline__ void nu3_mid_of(int id, const float* At, float* om, float* uz, int n, int lane, const Nu3Op op) {
#define MIX_TRI(k)                                                                              \
    case k:                                                                                     \
        if constexpr (tri_l(k).l1 <= L) nu3_mid<k, NP, QB, TCM>(At, om, uz, n, lane, op);       \
        break;
    switch (id) {
        MIX_TRI(0) MIX_TRI(1) MIX_TRI(2) MIX_TRI(3) MIX_TRI(4) MIX_TRI(5) MIX_TRI(6) MIX_TRI(7) MIX_TRI(8) MIX_TRI(9)
        MIX_TRI(10) MIX_TRI(11) MIX_TRI(12) MIX_TRI(13) MIX_TRI(14) MIX_TRI(15) MIX_TRI(16) MIX_TRI(17) MIX_TRI(18)
        MIX_TRI(19) MIX_TRI(20) MIX_TRI(21) MIX_TRI(22) MIX_TRI(23) MIX_TRI(24) MIX_TRI(25) MIX_TRI(26) MIX_TRI(27)
        MIX_TRI(28) MIX_TRI(29)
    }
#undef MIX_TRI
}

}  // namespace mixd
