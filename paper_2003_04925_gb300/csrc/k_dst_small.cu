// Dirichlet Poisson solve of meshes up to 128^3 on the FP32 CUDA cores at FDA order 2: the plane
// passes of the dense FP32 form (App. C).
//
// With the x axis solved by elimination (k_dst_tri.cu) the z and y transforms of an x plane X
// are Y = S X S (S the symmetric sine matrix), forward and inverse alike, and a plane of Ng <= 128
// fits shared memory next to S and S X: one launch takes both transforms, three launches the
// solve (k_pm.cu's one-axis passes take five).  The dense FP32 form is the fastest where few or
// small boxes leave a solve bound by its launches, and its rounding error is about half that of
// the split tensor-core products: 8 boxes of 24^3 cells take 21 us a solve in these passes, 37 us
// in five and 32 us on the tensor cores (1 box of 48^3: 32, 53 and 35 us; 64 boxes of 48^3:
// 164, 386 and 105 us).
//
// A thread owns a 4 x 4 block of the plane: per step of the contraction two 16-byte shared loads
// feed 16 FMAs.  T = S X (contraction over rows: both operands are read along their rows), then
// Y = T S with T stored transposed by the same threads.
#include <algorithm>

#include "device_util.cuh"

namespace scola {

namespace {

constexpr int kSmallMaxN = 128;

// PAD: write the padded potential instead of a dense mesh.
template <bool PAD>
__global__ void __launch_bounds__(1024, 1)
k_dst_small(const BoxDesc *__restrict__ boxes, const DstTable *__restrict__ tables, const float *__restrict__ tab,
            const Chunk *__restrict__ items, int nitems, int npmax, const float *__restrict__ in,
            float *__restrict__ out) {
    extern __shared__ __align__(16) float sm[];
    float *S = sm, *X = sm + npmax * npmax, *Tt = X + npmax * npmax;   // rows of Np floats
    const int tid = threadIdx.x;
    int cur = -1;
    for (int it = blockIdx.x; it < nitems; it += gridDim.x) {
        const Chunk item = items[it];
        const BoxDesc &B = boxes[item.box];
        const int Ng = B.Ng, Np = (Ng + 3) & ~3, nt = Np / 4;
        __syncthreads();                                     // (the plane before is finished)
        if (B.tbl != cur) {
            cur = B.tbl;
            const DstTable T = tables[cur];
            for (int q = tid; q < Ng * Np; q += blockDim.x) S[q] = tab[T.st_off + (q / Np) * T.LS + q % Np];
        }
        const float *src = in + B.m_off + item.start * Ng * Ng;
        for (int q = tid; q < Ng * Np; q += blockDim.x) {
            const int j = q / Np, k = q - j * Np;
            X[q] = k < Ng ? src[j * Ng + k] : 0.0f;
        }
        __syncthreads();
        const int r = (tid / nt) * 4, c = (tid % nt) * 4;    // this thread's block
        float acc[4][4];
        auto product = [&](const float *a, const float *b) {
#pragma unroll
            for (int p = 0; p < 4; ++p)
#pragma unroll
                for (int q = 0; q < 4; ++q) acc[p][q] = 0.0f;
#pragma unroll 4
            for (int t = 0; t < Ng; ++t) {
                const float4 av = *reinterpret_cast<const float4 *>(a + t * Np + r);
                const float4 bv = *reinterpret_cast<const float4 *>(b + t * Np + c);
                const float ax[4] = {av.x, av.y, av.z, av.w}, bx[4] = {bv.x, bv.y, bv.z, bv.w};
#pragma unroll
                for (int p = 0; p < 4; ++p)
#pragma unroll
                    for (int q = 0; q < 4; ++q) acc[p][q] = fmaf(ax[p], bx[q], acc[p][q]);
            }
        };
        const bool own = tid < nt * nt;
        if (own) {
            product(S, X);                                   // T[r + p][c + q]
#pragma unroll
            for (int q = 0; q < 4; ++q)
                if (c + q < Ng)
                    *reinterpret_cast<float4 *>(Tt + (c + q) * Np + r) =
                        make_float4(acc[0][q], acc[1][q], acc[2][q], acc[3][q]);
        }
        __syncthreads();
        if (own) {
            product(Tt, S);                                  // Y[r + p][c + q]
            const int G = PAD ? B.gpad : 0, W = Ng + 2 * G;
            float *dst = out + (PAD ? B.pp_off : B.m_off) + ((item.start + G) * W + G) * W + G;
            const bool vec = (Ng & 3) == 0;                  // (interior rows start 16-byte aligned)
#pragma unroll
            for (int p = 0; p < 4; ++p) {
                if (r + p >= Ng) break;
                float *row = dst + (r + p) * W + c;
                if (vec) {
                    *reinterpret_cast<float4 *>(row) = make_float4(acc[p][0], acc[p][1], acc[p][2], acc[p][3]);
                } else {
#pragma unroll
                    for (int q = 0; q < 4; ++q)
                        if (c + q < Ng) row[q] = acc[p][q];
                }
            }
        }
    }
}

template <bool PAD>
cudaError_t run_small(Ctx &c, const float *in, float *out) {
    // (256 threads load the plane and S also where fewer own blocks of it: latency counts here)
    const int np = (c.max_ng + 3) & ~3, threads = std::max(256, ((np / 4) * (np / 4) + 31) / 32 * 32);
    const size_t smem = 3 * (size_t)np * np * sizeof(float);
    const int per = std::max(1, std::min(2048 / threads, (int)(220 * 1024 / (smem + 1024))));
    const bool one = c.view_box >= 0;
    const Chunk *items = c.xplanes + (one ? c.xplane_beg[c.view_box] : 0);
    const int n = one ? c.boxes_h[c.view_box].Ng : c.n_xplanes;
    k_dst_small<PAD><<<std::max(1, std::min(n, per * c.num_sms)), threads, smem, c.stream>>>(
        c.boxes, c.tables, c.table_arena, items, n, np, in, out);
    ++c.launches;
    return cudaGetLastError();
}

}  // namespace

cudaError_t init_small_kernels() {
    const int smem = 3 * kSmallMaxN * kSmallMaxN * (int)sizeof(float);
    cudaError_t e = cudaFuncSetAttribute(k_dst_small<false>, cudaFuncAttributeMaxDynamicSharedMemorySize, smem);
    if (e != cudaSuccess) return e;
    return cudaFuncSetAttribute(k_dst_small<true>, cudaFuncAttributeMaxDynamicSharedMemorySize, smem);
}

// The dense FP32 form takes the plane passes where every mesh fits and the order is 2.
bool small_supported(const Ctx &c) { return c.prm.fda_order == 2 && c.max_ng <= kSmallMaxN; }

cudaError_t launch_small_pass(Ctx &c, int pass, const float *in, float *w1, float *out_pad) {
    switch (pass) {
        case 0: return run_small<false>(c, in, w1);
        case 1: return launch_tri_pass(c, w1);
        case 2: return run_small<true>(c, w1, out_pad);
        default: return cudaSuccess;
    }
}

}  // namespace scola
