// Device helpers shared by the kernels.
#pragma once

#include "internal.h"

namespace scola {

// The padded PM grid of a box has P = 2 N_ghost = FDA order ghost layers on every side
// (padded index pc = c + P, S = Ng + 2P cells per axis).

// Number of padded cells outside the interior: (Ng+2P)^3 - Ng^3.
__host__ __device__ inline long long shell_count(int Ng, int P) {
    const long long a = Ng + 2 * P;
    return a * a * a - (long long)Ng * Ng * Ng;
}

// Padded coordinates (0..Ng+2P-1 per axis) of shell cell `idx`.  Enumeration: the 2P
// full i-planes {0..P-1, Ng+P..Ng+2P-1}; then, for interior i, the 2P full j-rows; then,
// for interior i and j, the 2P k-cells.  (32-bit arithmetic: a shell of Ng <= 256, P <= 6
// has fewer than 2^22 cells.)
__device__ inline void shell_coord(long long idx64, int Ng, int P, int &pi, int &pj, int &pk) {
    int idx = (int)idx64;
    const int S = Ng + 2 * P;
    const int plane = S * S;
    const int A = 2 * P * plane;
    if (idx < A) {
        const int q = idx / plane;
        const int r = idx - q * plane;
        pi = q < P ? q : Ng + q;
        pj = r / S;
        pk = r - pj * S;
        return;
    }
    idx -= A;
    const int rowblk = 2 * P * S;
    const int B = Ng * rowblk;
    if (idx < B) {
        pi = P + idx / rowblk;
        const int r = idx - (pi - P) * rowblk;
        const int q = r / S;
        pj = q < P ? q : Ng + q;
        pk = r - q * S;
        return;
    }
    idx -= B;
    const int line = 2 * P * Ng;
    pi = P + idx / line;
    const int r = idx - (pi - P) * line;
    pj = P + r / (2 * P);
    const int q = r - (pj - P) * (2 * P);
    pk = q < P ? q : Ng + q;
}

// Central-difference coefficients of FDA order 2, 4, 6 (N_ghost = order / 2 terms):
// gradient f' = (1/d) sum_m g_m (f_{+m} - f_{-m}); second derivative
// f'' = (1/d^2) (s_0 f + sum_m s_m (f_{+m} + f_{-m})).
template <int ORDER> struct Fda;
template <> struct Fda<2> {
    static constexpr int ng = 1;
    __device__ static float g(int m) { return 0.5f; }
    __device__ static float s(int m) { return m == 0 ? -2.0f : 1.0f; }
};
template <> struct Fda<4> {
    static constexpr int ng = 2;
    __device__ static float g(int m) { return m == 1 ? 2.0f / 3.0f : -1.0f / 12.0f; }
    __device__ static float s(int m) { return m == 0 ? -2.5f : (m == 1 ? 4.0f / 3.0f : -1.0f / 12.0f); }
};
template <> struct Fda<6> {
    static constexpr int ng = 3;
    __device__ static float g(int m) { return m == 1 ? 0.75f : (m == 2 ? -0.15f : 1.0f / 60.0f); }
    __device__ static float s(int m) {
        return m == 0 ? -49.0f / 18.0f : (m == 1 ? 1.5f : (m == 2 ? -0.15f : 1.0f / 90.0f));
    }
};

// Boundary term of Eq. 62 for the interior cell (i, j, k): the order-n Laplacian's
// contributions of the Dirichlet values in the ghost layers (unscaled by 1/dg^2).  P_c is
// the padded potential at the cell; S the padded row length.  Per axis: the offsets m
// that reach past the lower face (m > x) and past the upper face (m >= Ng - x).
template <int ORDER>
__device__ __forceinline__ float boundary_term_n(const float *P_c, int i, int j, int k, int Ng, int S) {
    float bc = 0.0f;
    const int st[3] = {S * S, S, 1};
    const int x[3] = {i, j, k};
#pragma unroll
    for (int a = 0; a < 3; ++a) {
#pragma unroll
        for (int m = 1; m <= Fda<ORDER>::ng; ++m) {
            if (m > x[a]) bc += Fda<ORDER>::s(m) * P_c[-m * st[a]];
            if (m >= Ng - x[a]) bc += Fda<ORDER>::s(m) * P_c[m * st[a]];
        }
    }
    return bc;
}

__device__ __forceinline__ float boundary_term(const float *P_c, int i, int j, int k, int Ng, int S, int order) {
    return order == 2 ? boundary_term_n<2>(P_c, i, j, k, Ng, S)
                      : (order == 4 ? boundary_term_n<4>(P_c, i, j, k, Ng, S) : boundary_term_n<6>(P_c, i, j, k, Ng, S));
}

// Quotient and remainder of v / n for 0 <= v < n^3 < 2^31, from a reciprocal.  The conversion of v,
// the reciprocal (2 ulp) and the product are off by less than 2^-21.4 together, of a quotient
// below 2^20.7: less than one, so one step of correction on the exact integer remainder is enough.
// (Each particle kernel decodes its lattice site with two of these; with integer divisions, and a
// clearing pass in the atomic deposit: 21 evaluations of 64 boxes of 48^3 particles 16.90 ms, now
// 16.67; one force evaluation on 64 boxes of 96^3 cells 826 us, now 816.)
__device__ __forceinline__ int div_small(int v, int n, float inv, int &rem) {
    int q = __float2int_rz((float)v * inv);
    rem = v - q * n;
    if (rem >= n) {
        rem -= n;
        ++q;
    } else if (rem < 0) {
        rem += n;
        --q;
    }
    return q;
}

__device__ __forceinline__ void decode_local(int local, int n, int &i, int &j, int &k) {
    const float inv = __fdividef(1.0f, (float)n);
    i = div_small(div_small(local, n, inv, k), n, inv, j);
}

// Blocks of 256 lattice sites for the kernels that gather from the mesh: 4 x (64 / z) x z sites
// (x, y, z extents), z = 16 where that divides the box, else 8.  A block's stencils share more
// cache lines than a run of 256 sites along z, and its state is still read in whole sectors.
// Boxes that blocks would cover with more than an eighth of idle lanes (25 sites a side: 83 %)
// keep the runs: block_z = 0.
__host__ __device__ inline int block_tiles(int Nsc, int bz) {
    const int sy = bz == 16 ? 2 : 3, sz = bz == 16 ? 4 : 3;
    return ((Nsc + 3) >> 2) * ((Nsc + (1 << sy) - 1) >> sy) * ((Nsc + bz - 1) >> sz);
}
__host__ __device__ inline int block_z(int Nsc) {
    const int bz = (Nsc & 15) == 0 ? 16 : 8;
    return 8LL * 256 * block_tiles(Nsc, bz) <= 9LL * Nsc * Nsc * Nsc ? bz : 0;
}
__host__ __device__ inline int block_count(int Nsc) {
    const int bz = block_z(Nsc);
    return bz ? block_tiles(Nsc, bz) : (Nsc * Nsc * Nsc + 255) / 256;
}
// Site t (0 .. 255) of block q of a box; false beyond the lattice.
__device__ __forceinline__ bool block_site(int q, int t, int Nsc, int &i, int &j, int &k) {
    const int bz = block_z(Nsc);
    if (bz == 0) {
        decode_local(q * 256 + t, Nsc, i, j, k);
        return i < Nsc;
    }
    const int sy = bz == 16 ? 2 : 3, sz = bz == 16 ? 4 : 3;
    const int nz = (Nsc + bz - 1) >> sz, ny = (Nsc + (1 << sy) - 1) >> sy;
    int bj, bk;
    const int r = div_small(q, nz, __fdividef(1.0f, (float)nz), bk);
    i = (div_small(r, ny, __fdividef(1.0f, (float)ny), bj) << 2) + (t >> 6);
    j = (bj << sy) + ((t & 63) >> sz);
    k = (bk << sz) + (t & (bz - 1));
    return i < Nsc && j < Nsc && k < Nsc;
}

// Per-tile final scale factors: box b's FP32 coefficients at force evaluation k (see Ctx::coef),
// or null when the launch uses uniform scalars.
__device__ __forceinline__ const float *box_coef(const float *coef, int box, int k, int nk) {
    return coef ? coef + ((long long)box * nk + k) * 8 : nullptr;
}

// Sorted deposit: the interior mesh of a box is cut into bricks of kBrick^3 cells.
constexpr int kBrick = 16;

struct SortEntry {
    int key;          // box-local key ((bx nbe + by) nbe + bz) 8 + class, or -1 (no weight inside)
    float4 e;         // f_x, f_y, f_z, packed i0 (+2, 10 bits per axis)
};

// The sorted deposit's key and entry of a particle at box-local lattice index b with
// displacement s: the clamped mesh coordinate u (as in the CIC deposit) has integer part
// i0 and fractions f; the key is the brick of the upper corner i0 + 1 with a 3-bit class
// whose bit a says that the lower corner lies in the brick below along axis a.  The count
// pass (in the kick-drift of the previous step, or its own kernel) and the fill pass
// compute it with this one function from the same FP32 values.
__device__ __forceinline__ SortEntry brick_entry(const BoxDesc &B, const float (&s)[3], const int (&b)[3]) {
    const int Ng = B.Ng, nbe = B.nbe;
    int i0[3];
    float f[3];
    bool inside = true;
#pragma unroll
    for (int a = 0; a < 3; ++a) {
        float u = fmaf(s[a], B.inv_dg, fmaf((float)b[a], B.q2u, 0.5f * B.q2u - 0.5f));
        u = fminf(fmaxf(u, -2.0f), (float)Ng + 1.0f);
        const float fl = floorf(u);
        i0[a] = (int)fl;
        f[a] = u - fl;
        inside = inside && i0[a] >= -1 && i0[a] < Ng;
    }
    SortEntry r;
    r.key = -1;
    r.e = make_float4(f[0], f[1], f[2],
                      __int_as_float((i0[0] + 2) | ((i0[1] + 2) << 10) | ((i0[2] + 2) << 20)));
    if (inside) {
        const int cls = (((i0[0] + 1) & (kBrick - 1)) == 0 ? 1 : 0) | (((i0[1] + 1) & (kBrick - 1)) == 0 ? 2 : 0) |
                        (((i0[2] + 1) & (kBrick - 1)) == 0 ? 4 : 0);
        r.key = ((((i0[0] + 1) >> 4) * nbe + ((i0[1] + 1) >> 4)) * nbe + ((i0[2] + 1) >> 4)) * 8 + cls;
    }
    return r;
}

// 2^-32 fixed-point value of a CIC weight w in [0, 1]: round-to-nearest of w 2^32 (the
// same integer as a direct float -> uint64 conversion), computed with 32-bit conversions
// only (64-bit integer conversions run on the FP64 pipe, which is narrow on this GPU).
__device__ __forceinline__ unsigned long long weight_to_fixed(float w) {
    const float v = w * 4294967296.0f;
    return v >= 4294967296.0f ? (1ull << 32) : (unsigned long long)__float2uint_rn(v);
}

// Correctly rounded float of a 64-bit count (round to nearest even, as a direct
// uint64 -> float conversion), from 32-bit operations: the top 32 significant bits with a
// sticky bit for the rest, converted once and scaled by an exact power of two.
__device__ __forceinline__ float fixed_to_float(unsigned long long x) {
    const unsigned hi = (unsigned)(x >> 32), lo = (unsigned)x;
    if (hi == 0) return __uint2float_rn(lo);
    const int lz = __clz(hi);
    const unsigned top = lz ? (hi << lz) | (lo >> (32 - lz)) : hi;
    const unsigned rest = lz ? lo << lz : lo;
    const float m = __uint2float_rn(top | (rest != 0u ? 1u : 0u));
    return m * __int_as_float((127 + 32 - lz) << 23);
}

// Trilinear stencil on the LPT grid (nodes at (i + 1/2) dq, N = Np) at the centre of padded
// mesh cell pc of a box (C.3): lower node i0 (not wrapped) and offsets f.  In node units the
// cell centre is u = (t Ntile - Nbuf) + ((2 pc - 3) Nsc - Ng) / (2 Ng), so i0 and the
// remainder are exact integers and f is one correctly rounded division.
__device__ __forceinline__ void shell_stencil(const BoxDesc &B, const int pc[3], int Ntile, int i0[3], float f[3]) {
    const int t[3] = {B.tx, B.ty, B.tz};
    const int den = 2 * B.Ng;
#pragma unroll
    for (int a = 0; a < 3; ++a) {
        const int num = (2 * (pc[a] - B.gpad) + 1) * B.Nsc - B.Ng;
        int q = num / den, r = num - q * den;
        if (r < 0) {
            r += den;
            --q;
        }
        i0[a] = t[a] * Ntile - B.Nbuf + q;
        f[a] = (float)r / (float)den;
    }
}

// The same stencil with each offset as the exact remainder r of r / (2 Ng).
__device__ __forceinline__ void shell_stencil_r(const BoxDesc &B, const int pc[3], int Ntile, int i0[3], int rem[3]) {
    const int t[3] = {B.tx, B.ty, B.tz};
    const int den = 2 * B.Ng;
#pragma unroll
    for (int a = 0; a < 3; ++a) {
        const int num = (2 * (pc[a] - B.gpad) + 1) * B.Nsc - B.Ng;
        int q = num / den, r = num - q * den;
        if (r < 0) {
            r += den;
            --q;
        }
        i0[a] = t[a] * Ntile - B.Nbuf + q;
        rem[a] = r;
    }
}

// Unevaluated sums h + l of two floats (about 47 significant bits), for the C.3 shell where they
// decide its rounding: FP64 runs at 1/64 of the FP32 rate on this GPU.  Sums by Knuth's two-sum, products by one FMA remainder
// (Dekker 1971, Knuth TAOCP vol. 2, 4.2.2); the _rn intrinsics keep the compiler from fusing.
struct FloatPair {
    float h, l;
};

__device__ __forceinline__ FloatPair two_sum(float a, float b) {
    const float s = __fadd_rn(a, b), t = __fsub_rn(s, a);
    return {s, __fadd_rn(__fsub_rn(a, __fsub_rn(s, t)), __fsub_rn(b, t))};
}

// a + f (b - a)
__device__ __forceinline__ FloatPair pair_lerp(FloatPair a, FloatPair b, FloatPair f) {
    FloatPair d = two_sum(b.h, -a.h);
    d.l = __fadd_rn(d.l, __fsub_rn(b.l, a.l));
    const float th = __fmul_rn(f.h, d.h);
    const float tl = __fmaf_rn(f.l, d.h, __fmaf_rn(f.h, d.l, __fmaf_rn(f.h, d.h, -th)));
    FloatPair r = two_sum(a.h, th);
    r.l = __fadd_rn(r.l, __fadd_rn(a.l, tl));
    const float h = __fadd_rn(r.h, r.l);
    return {h, __fsub_rn(r.l, __fsub_rn(h, r.h))};
}

// Whether every value within e of x.h + x.l rounds to x.h (false for infinities and NaN).
__device__ __forceinline__ bool pair_rounds(FloatPair x, float e) {
    return __fadd_rn(x.h, __fadd_rn(x.l, e)) == x.h && __fadd_rn(x.h, __fsub_rn(x.l, e)) == x.h;
}

__device__ __forceinline__ int wrap(int v, int n) {
    v %= n;
    return v < 0 ? v + n : v;
}

// The same for v within one period of [0, n) (indices next to a position in the box): a compare
// and an add; anything further out takes the remainder.
__device__ __forceinline__ int wrap_near(int v, int n) {
    if (v < 0) v += n;
    if (v >= n) v -= n;
    return (unsigned)v < (unsigned)n ? v : wrap(v, n);
}

// Periodic CIC deposit of one particle per lane on an N^3 grid of 2^-32 fixed-point counts: lower
// corner i0 (not wrapped), fractions f; every lane of the warp calls it (valid or not).
// kMerge, for grids of one cell per particle spacing: consecutive lanes hold Lagrangian
// z-neighbours, and where a lane's lower corner is its left neighbour's moved one cell up in z the
// neighbour's four upper-z weights join its own lower-z ones and the neighbour skips those atomics
// (integer sums: the same totals).
template <bool kMerge>
__device__ __forceinline__ void periodic_deposit(unsigned long long *acc, int N, const int (&i0)[3], const float (&f)[3],
                                                 bool valid) {
    bool take = false, give = false;
    if (kMerge) {
        const int lane = threadIdx.x & 31, key = valid ? i0[2] : 0x40000000;
        const int px = __shfl_up_sync(0xffffffffu, i0[0], 1), py = __shfl_up_sync(0xffffffffu, i0[1], 1),
                  pz = __shfl_up_sync(0xffffffffu, key, 1);
        take = valid && lane > 0 && px == i0[0] && py == i0[1] && pz + 1 == i0[2];
        give = __shfl_down_sync(0xffffffffu, take ? 1 : 0, 1) && lane < 31;
    }
    const int z0 = wrap_near(i0[2], N), z1 = z0 + 1 == N ? 0 : z0 + 1;
#pragma unroll
    for (int dx = 0; dx < 2; ++dx) {
        const float wx = dx ? f[0] : 1.0f - f[0];
#pragma unroll
        for (int dy = 0; dy < 2; ++dy) {
            const float wxy = wx * (dy ? f[1] : 1.0f - f[1]);
            unsigned long long lo = weight_to_fixed(wxy * (1.0f - f[2])), up = weight_to_fixed(wxy * f[2]);
            if (kMerge) {
                const unsigned long long left = __shfl_up_sync(0xffffffffu, up, 1);
                if (take) lo += left;
            }
            if (!valid) continue;
            unsigned long long *row = acc + ((long long)wrap_near(i0[0] + dx, N) * N + wrap_near(i0[1] + dy, N)) * N;
            atomicAdd(row + z0, lo);
            if (!give) atomicAdd(row + z1, up);
        }
    }
}

}  // namespace scola
