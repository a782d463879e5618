// Dirichlet Poisson solve at FDA order 2: the x axis by elimination (App. C).
//
// After the DST-I along z and y, the order-2 Laplacian is tridiagonal along x for every pair of
// frequencies (m, n): dividing the x transform by lambda_l + lambda_m + lambda_n and transforming
// back (Eq. 71) solves exactly
//   (2 + mu) u_i - u_{i-1} - u_{i+1} = -dg^2 f_i,  u = 0 on the two Dirichlet planes,
//   mu = -dg^2 (lambda_m + lambda_n) = 4 (sin^2 t_m + sin^2 t_n),  t_m = pi m / (2 (Ng + 1)),
// so one forward and one backward recursion take the place of two dense transforms: the solve
// needs four one-axis transforms (or two plane passes of two) and this pass, which moves each
// cell once in and once out.  With c_i the inverse pivots,
//   y_i = c_i (kappa f_i + y_{i-1}),  u_i = y_i + c_i u_{i+1},  c_i = 1 / (2 + mu - c_{i-1}),
// every coefficient is positive (no cancellation: the recursions are as accurate as the
// transforms they replace).  1 - c_i is what the pivots carry (c_i = 1 / (1 + h), 1 - c_i = h c_i,
// h = mu + 1 - c_{i-1}), so that mu keeps its relative accuracy next to 1 at low frequencies.
// The elimination runs from both planes at once (the right half by symmetry uses the same
// pivots) and meets in the middle, at rows a = ceil(Ng / 2) and a + 1:
//   u_a = (y_a + c_a z_{a+1}) / (1 - c_a c_b),  u_{a+1} = z_{a+1} + c_b u_a,  b = Ng - a,
// which halves the chains and doubles the threads for the same shared memory.
// kappa = -dg^2 (2 / (Ng + 1))^2 also holds the scale of the two inverse transforms.
//
// A pair of threads owns one column (m, n) of one box: consecutive threads read and write
// consecutive floats of every x plane, and columns never meet.  A CTA takes 64 columns of several
// boxes at a time and walks the boxes of its column tile; the pivots depend on the column alone
// and are computed once per tile.  y waits in shared memory for the backward recursion (this is
// what bounds the resident threads), the next rows of f, also those of the next boxes, are in
// flight in registers: 8 rows up to Ng = 128 (two CTAs of 512 threads an SM for four or more boxes
// of 96^3), 16 above, where fewer threads fit (16 boxes of 192^3: 290 us with 8 rows, 214 us with
// 16; 64 of 96^3: 106 us and 112 us).  Bound: HBM, 8 bytes a cell.
#include <algorithm>
#include <cstring>
#include <vector>

#include "device_util.cuh"

namespace scola {

namespace {

constexpr int kTriW = 64;            // columns per CTA and box
constexpr int kTriParts = 4;         // boxes side by side in a CTA, at most
constexpr int kTriGroups = 4;
constexpr size_t kTriSmem = 227 * 1024;

struct TriGroupArgs {
    const Chunk *items;              // the group's boxes
    const float *mu;                 // 4 sin^2 t_l, Ng
    float kappa;
    int nboxes, Ng, cta0, nctas;
};

struct TriArgs {
    TriGroupArgs grp[kTriGroups];
    int ngroups;
    const BoxDesc *boxes;
    float *mesh;
};

// kTriB: rows of f in flight per thread.
template <int kTriB>
__global__ void __launch_bounds__(2 * kTriW * kTriParts) k_dst_tri(const __grid_constant__ TriArgs A) {
    extern __shared__ __align__(16) float sm[];
    int gi = 0;
    while (gi + 1 < A.ngroups && (int)blockIdx.x >= A.grp[gi + 1].cta0) ++gi;
    const TriGroupArgs &G = A.grp[gi];
    const int Ng = G.Ng, Ng2 = Ng * Ng, nb = G.nboxes, half = (Ng + 1) / 2;
    const int lane = threadIdx.x & (kTriW - 1), side = (threadIdx.x / kTriW) & 1, part = threadIdx.x / (2 * kTriW);
    const int parts = blockDim.x / (2 * kTriW);
    const int n = side ? Ng - half : half;                  // rows of this thread, from its plane inwards
    // items of the group: (column tile, `parts` boxes), the boxes of a tile in turn; this CTA
    // takes a contiguous range
    const int per = (nb + parts - 1) / parts;
    const long long total = (long long)((Ng2 + kTriW - 1) / kTriW) * per;
    const int cta = (int)blockIdx.x - G.cta0;
    const long long lo = total * cta / G.nctas, hi = total * (cta + 1) / G.nctas;
    // shared memory: pivots [half][W], 1 / (1 - c_a c_b) [W], the meeting rows' y of two
    // consecutive items [2][parts][2][W], y [parts][2][half][W]
    float *cs = sm + lane, *inv = cs + half * kTriW, *meet = inv + kTriW + 2 * part * kTriW;
    float *ys = sm + (half + 1 + 4 * parts) * kTriW + (2 * part + side) * half * kTriW + lane;
    // this thread's first row in its column of item q, or null beyond the mesh or the group's boxes
    auto column = [&](long long q) -> float * {
        if (q >= hi) return nullptr;
        const int tile = (int)(q / per), box = (int)(q - (long long)tile * per) * parts + part;
        const int col = tile * kTriW + lane;
        if (box >= nb || col >= Ng2) return nullptr;
        return A.mesh + A.boxes[G.items[box].box].m_off + col + (side ? (Ng - 1) * Ng2 : 0);
    };
    const int step = side ? -Ng2 : Ng2;
    float xn[kTriB];
    auto fetch = [&](const float *src, int k0) {
#pragma unroll
        for (int j = 0; j < kTriB; ++j) xn[j] = src && k0 + j < n ? src[(k0 + j) * step] : 0.0f;
    };
    float *mine = column(lo);
    fetch(mine, 0);
    int cur = -1;
    for (long long q = lo; q < hi; ++q) {
        const int tile = (int)(q / per);
        if (tile != cur) {                                  // (the same for the whole CTA)
            cur = tile;
            const int col = tile * kTriW + lane;
            __syncthreads();
            if (threadIdx.x < kTriW && col < Ng2) {
                const float mu = G.mu[col / Ng] + G.mu[col % Ng];
                float g = 1.0f, gb = 1.0f;                  // 1 - c of the row before; of row b
                for (int k = 0; k < half; ++k) {
                    const float h = mu + g, c = 1.0f / (1.0f + h);
                    cs[k * kTriW] = c;
                    g = h * c;
                    if (k == Ng - half - 1) gb = g;
                }
                *inv = 1.0f / (g + gb - g * gb);
            }
            __syncthreads();
        }
        float *next = column(q + 1);
        float y = 0.0f;
        for (int k0 = 0; k0 < n; k0 += kTriB) {
            float cv[kTriB], tv[kTriB];
#pragma unroll
            for (int j = 0; j < kTriB; ++j) {
                cv[j] = k0 + j < n ? cs[(k0 + j) * kTriW] : 0.0f;
                tv[j] = cv[j] * (G.kappa * xn[j]);
            }
            if (k0 + kTriB < n) fetch(mine, k0 + kTriB);
            else fetch(next, 0);
#pragma unroll
            for (int j = 0; j < kTriB; ++j)
                if (k0 + j < n) {
                    y = fmaf(cv[j], y, tv[j]);
                    ys[(k0 + j) * kTriW] = y;
                }
        }
        // the meeting rows (slots alternate between items: a thread is at most one item ahead)
        float *mt = meet + (int)((q - lo) & 1) * 2 * parts * kTriW;
        mt[side * kTriW] = y;
        __syncthreads();
        if (mine && n > 0) {                                // (a mesh of one cell has no second half)
            const float ua = fmaf(cs[(half - 1) * kTriW], mt[kTriW], mt[0]) * *inv;
            float u = side ? fmaf(cs[(n - 1) * kTriW], ua, mt[kTriW]) : ua;     // (row b = n - 1 there)
            mine[(n - 1) * step] = u;
            for (int k0 = n - 2; k0 >= 0; k0 -= kTriB) {
                float cv[kTriB], yv[kTriB];
#pragma unroll
                for (int j = 0; j < kTriB; ++j) {
                    cv[j] = k0 - j >= 0 ? cs[(k0 - j) * kTriW] : 0.0f;
                    yv[j] = k0 - j >= 0 ? ys[(k0 - j) * kTriW] : 0.0f;
                }
#pragma unroll
                for (int j = 0; j < kTriB; ++j) {
                    u = fmaf(cv[j], u, yv[j]);
                    if (k0 - j >= 0) mine[(k0 - j) * step] = u;
                }
            }
        }
        mine = next;
    }
}

size_t tri_smem(int Ng, int parts) {
    const size_t half = (Ng + 1) / 2;
    return (half + 1 + 4 * parts + 2 * parts * half) * kTriW * sizeof(float);
}

}  // namespace

cudaError_t init_tri_kernel() {
    for (const void *f : {(const void *)k_dst_tri<8>, (const void *)k_dst_tri<16>}) {
        cudaError_t e = cudaFuncSetAttribute(f, cudaFuncAttributeMaxDynamicSharedMemorySize, (int)kTriSmem);
        if (e == cudaSuccess)
            e = cudaFuncSetAttribute(f, cudaFuncAttributePreferredSharedMemoryCarveout, cudaSharedmemCarveoutMaxShared);
        if (e != cudaSuccess) return e;
    }
    return cudaSuccess;
}

// In place on the meshes [i][m][n] (x, y frequency, z frequency) of every box of the view.
cudaError_t launch_tri_pass(Ctx &c, float *mesh) {
    std::vector<TriGroupArgs> all;
    for (const TriGroup &T : c.tri_groups) {
        TriGroupArgs P;
        P.Ng = T.Ng;
        P.items = T.boxes;
        P.nboxes = T.nboxes;
        if (c.view_box >= 0) {
            if (c.boxes_h[c.view_box].Ng != T.Ng) continue;
            P.items = c.tri_boxes + c.tri_box_at[c.view_box];
            P.nboxes = 1;
        }
        if (P.nboxes < 1) continue;                          // (a batch may hold no box of an Ng)
        P.mu = c.table_arena + T.mu_off;
        P.kappa = T.kappa;
        all.push_back(P);
    }
    for (size_t g0 = 0; g0 < all.size(); g0 += kTriGroups) {
        const int ng = (int)std::min(all.size() - g0, (size_t)kTriGroups);
        TriArgs a;
        std::memset(&a, 0, sizeof(a));
        int ngmax = 0, nbmax = 1;
        double total = 0;
        std::vector<double> work(ng);
        for (int g = 0; g < ng; ++g) {
            const TriGroupArgs &P = a.grp[g] = all[g0 + g];
            work[g] = (double)P.Ng * P.Ng * P.Ng * P.nboxes;
            total += work[g];
            ngmax = std::max(ngmax, P.Ng);
            nbmax = std::max(nbmax, P.nboxes);
        }
        // boxes side by side in a CTA: the number that keeps most threads resident per SM (four boxes
        // or more of 96^3: 4, in 2 CTAs; of 192^3: 4, in 1 CTA; two or three of 96^3: 2, in 3 CTAs)
        int parts = 1, ctas = 1;
        for (int p = 1; p <= kTriParts && p <= nbmax; ++p) {
            const int n = std::min(16 / p, (int)(kTriSmem / (tri_smem(ngmax, p) + 1024)));
            if (n * p > parts * ctas || p == 1) parts = p, ctas = std::max(1, n);
        }
        // the grid is one wave, split among the groups in proportion to their cells
        const int slots = c.num_sms * ctas;
        int cta0 = 0;
        for (int g = 0; g < ng; ++g) {
            TriGroupArgs &P = a.grp[g];
            const long long items = ((long long)P.Ng * P.Ng + kTriW - 1) / kTriW * ((P.nboxes + parts - 1) / parts);
            P.cta0 = cta0;
            P.nctas = (int)std::max(1LL, std::min(items, (long long)(slots * work[g] / std::max(total, 1.0))));
            cta0 += P.nctas;
        }
        a.ngroups = ng;
        a.boxes = c.boxes;
        a.mesh = mesh;
        if (ngmax <= 128) k_dst_tri<8><<<cta0, 2 * kTriW * parts, tri_smem(ngmax, parts), c.stream>>>(a);
        else k_dst_tri<16><<<cta0, 2 * kTriW * parts, tri_smem(ngmax, parts), c.stream>>>(a);
        ++c.launches;
        const cudaError_t e = cudaGetLastError();
        if (e != cudaSuccess) return e;
    }
    return cudaSuccess;
}

}  // namespace scola
