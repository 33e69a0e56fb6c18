// kernels_mean.cu -- the mean step of Alg. 1 on sm_103a:
//   step 1   zbar = argmin_z sum_k ||y_k - A_k z||^2, by conjugate gradients on
//            the normal equations A^H A z = A^H y (CGLS) from z = 0;
//   step 2a  y~_k = y_k - A_k zbar.
// The normal operator A^H A = sum_k A_k^H A_k is the iteration's transform
// pipeline at rank 1 with b_k = 1 (launch_normal_op in kernels_iter.cu): with
// line masks it is sum_j conj(d_j) o F_y^H[c_ky F_y(d_j o z)], c_ky the number
// of frames that sample row ky.  This file holds the right-hand side, one CG
// step and the residual pass.
//
// CG vectors live in the context's n x r buffers (first column): p in U (the
// operator's input), A^H A p in U+ (its output), z in U_{t-1}, s = A^H r in
// the gradient buffer.  The CG scalars are FP64, summed in a fixed order.
#include <math.h>

#include <algorithm>

#include "common.cuh"
#include "fft.cuh"
#include "internal.h"

#define CG_THREADS 256

// The vectors (n complex values, L2 resident) are spread over every
// multiprocessor and the FP64 scalars close each kernel: the last block to
// arrive adds the blocks' partial sums in block order and forms the next
// scalar, so a CG step is three short launches.  192 x 192, q = 48, kernel time,
// one block of 1024 threads -> this form: right-hand side 868 -> 20 us,
// one CG step 141 -> 15 us (the sum of its three kernels).

// Sum over the block of one FP64 value per thread: warp shuffles, then the
// warps in order (deterministic); valid in thread 0.
static __device__ double block_sum_fp64(double v) {
    __shared__ double red[CG_THREADS / 32];
    v = warp_sum_d(v);
    if ((threadIdx.x & 31) == 0) red[threadIdx.x >> 5] = v;
    __syncthreads();
    double t = 0.0;
    if (threadIdx.x == 0)
        for (int w = 0; w < CG_THREADS / 32; ++w) t += red[w];
    return t;
}

// Grid-wide sum of one FP64 value per thread: true in the first warp of the
// last block, where `total` is the sum of the blocks' partials (lane-strided,
// then a fixed shuffle tree).
static __device__ bool grid_sum_fp64(double v, double *part, unsigned int *counter, double &total) {
    const double b = block_sum_fp64(v);
    if (threadIdx.x == 0) part[blockIdx.x] = b;
    if (!last_block_arrive(counter) || threadIdx.x >= 32) return false;
    double t = 0.0;
    for (int i = threadIdx.x; i < (int)gridDim.x; i += 32) t += __ldcg(part + i);
    total = warp_sum_d(t);
    return true;
}

// s = A^H y = sum_k Z[:, k] (Z = [A_k^H y_k], row-major i q + k), p = s, z = 0,
// B = 1 (q x 1); cg = {||s||^2, 0, 0, 0}.  One warp per pixel.
__global__ void __launch_bounds__(CG_THREADS) k_cg_init(const float2 *__restrict__ Z, int n, int q, float2 *s,
                                                        float2 *p, float2 *z, float2 *B, double *cg, double *part,
                                                        unsigned int *counter) {
    const int lane = threadIdx.x & 31, warps = gridDim.x * (CG_THREADS / 32);
    double acc = 0.0;
    for (int i = blockIdx.x * (CG_THREADS / 32) + (threadIdx.x >> 5); i < n; i += warps) {
        float2 v = make_float2(0.f, 0.f);
        for (int k = lane; k < q; k += 32) v = cadd(v, __ldg(Z + (size_t)i * q + k));
#pragma unroll
        for (int o = 16; o > 0; o >>= 1) v = cadd(v, shfl_xor2(v, o));
        if (lane == 0) {
            s[i] = v;
            p[i] = v;
            z[i] = make_float2(0.f, 0.f);
            acc += (double)v.x * v.x + (double)v.y * v.y;
        }
    }
    if (blockIdx.x == 0)
        for (int k = threadIdx.x; k < q; k += blockDim.x) B[k] = make_float2(1.f, 0.f);
    double g;
    if (grid_sum_fp64(acc, part, counter, g) && lane == 0) {
        cg[0] = g;
        cg[1] = cg[2] = cg[3] = 0.0;
    }
}

// One CG step on A^H A z = A^H y, given w = A^H A p, in three kernels:
//   k_cg_dot    alpha = gamma / <p, w>
//   k_cg_update z += alpha p;  s -= alpha w;  gamma' = ||s||^2;  beta = gamma' / gamma
//   k_cg_dir    p = s + beta p
// cg = {gamma, alpha, stop, beta}: stop = 1 (and nothing updated) when <p, w> <= 0.
__global__ void __launch_bounds__(CG_THREADS) k_cg_dot(const float2 *__restrict__ p, const float2 *__restrict__ w, int n,
                                                       double *cg, double *part, unsigned int *counter) {
    double acc = 0.0;
    for (int i = blockIdx.x * CG_THREADS + threadIdx.x; i < n; i += gridDim.x * CG_THREADS) {
        const float2 a = p[i], b = w[i];
        acc += (double)a.x * b.x + (double)a.y * b.y;   // Re(conj(p_i) w_i)
    }
    double dot;
    if (grid_sum_fp64(acc, part, counter, dot) && threadIdx.x == 0) {
        if (dot > 0.0 && cg[0] > 0.0) cg[1] = cg[0] / dot;
        else cg[2] = 1.0;
    }
}
__global__ void __launch_bounds__(CG_THREADS) k_cg_update(const float2 *__restrict__ p, const float2 *__restrict__ w,
                                                          float2 *z, float2 *s, int n, double *cg, double *part,
                                                          unsigned int *counter) {
    if (cg[2] != 0.0) return;   // the same for every thread of the grid
    const float alpha = (float)cg[1];
    const double gamma = cg[0];
    double acc = 0.0;
    for (int i = blockIdx.x * CG_THREADS + threadIdx.x; i < n; i += gridDim.x * CG_THREADS) {
        const float2 a = p[i], b = w[i];
        float2 zz = z[i], ss = s[i];
        zz.x = fmaf(alpha, a.x, zz.x);
        zz.y = fmaf(alpha, a.y, zz.y);
        ss.x = fmaf(-alpha, b.x, ss.x);
        ss.y = fmaf(-alpha, b.y, ss.y);
        z[i] = zz;
        s[i] = ss;
        acc += (double)ss.x * ss.x + (double)ss.y * ss.y;
    }
    double g2;
    if (grid_sum_fp64(acc, part, counter, g2) && threadIdx.x == 0) {   // every block has read cg[0]
        cg[0] = g2;
        cg[3] = g2 / gamma;
    }
}
__global__ void __launch_bounds__(CG_THREADS) k_cg_dir(float2 *p, const float2 *__restrict__ s, int n,
                                                       const double *__restrict__ cg) {
    if (cg[2] != 0.0) return;
    const float beta = (float)cg[3];
    for (int i = blockIdx.x * CG_THREADS + threadIdx.x; i < n; i += gridDim.x * CG_THREADS) {
        const float2 ss = s[i], a = p[i];
        p[i] = make_float2(fmaf(beta, a.x, ss.x), fmaf(beta, a.y, ss.y));
    }
}

// y~ = y - A z on every sampled line.  T holds F_y(d_j o z) on the sampled rows
// (rank 1: T[(j ny + ky) nx + x]).  Row rr = j nl_k + i of frame k (coil j,
// line i, ky = framerows[lp_k + i]) is y[(C lp_k + rr) nx + kx]; the pass
// applies F_x (unitary) to T_j[ky, :] and subtracts.  Grid (ceil(C nl_max / 8), q).
template <int P>
__global__ void __launch_bounds__(256) k_mean_resid(const float2 *__restrict__ y, const float2 *__restrict__ T,
                                                     const int32_t *__restrict__ framerows,
                                                     const int32_t *__restrict__ lineptr, float2 *__restrict__ ytil,
                                                     int ny, int nc, const float2 *__restrict__ g_tw, float scale) {
    constexpr int N = 32 * P;
    constexpr int ROWS = 8, TPR = ROWS + 1;
    __shared__ float2 s_tw[N];
    __shared__ float2 tile[N * TPR];
    const int k = blockIdx.y;
    const int lp = lineptr[k], nl = lineptr[k + 1] - lp;
    const int rows_k = nc * nl;
    const int r0 = blockIdx.x * ROWS;
    if (r0 >= rows_k) return;   // the same for every thread of the block
    load_twiddles(s_tw, g_tw, N);
    for (int e = threadIdx.x; e < ROWS * N; e += blockDim.x) {
        const int row = e / N, x = e - row * N;
        const int rr = r0 + row;
        float2 a = make_float2(0.f, 0.f);
        if (rr < rows_k) {
            const int j = rr / nl, i = rr - j * nl;
            const int ky = framerows[lp + i];
            a = T[((size_t)j * ny + ky) * N + x];
        }
        tile[x * TPR + row] = a;
    }
    __syncthreads();
    fft::tile_dft<N, false>(tile, TPR, ROWS, s_tw, scale);
    for (int e = threadIdx.x; e < ROWS * N; e += blockDim.x) {
        const int row = e / N, kx = e - row * N;
        const int rr = r0 + row;
        if (rr < rows_k) {
            const size_t off = ((size_t)nc * lp + rr) * N + kx;
            const float2 a = y[off], b = tile[kx * TPR + row];
            ytil[off] = make_float2(a.x - b.x, a.y - b.y);
        }
    }
}

#define DISPATCH_P(PV, ...)                                           \
    switch (PV) {                                                      \
        case 1: { constexpr int P_ = 1; __VA_ARGS__; } break;                 \
        case 2: { constexpr int P_ = 2; __VA_ARGS__; } break;                 \
        case 3: { constexpr int P_ = 3; __VA_ARGS__; } break;                 \
        case 4: { constexpr int P_ = 4; __VA_ARGS__; } break;                 \
        case 5: { constexpr int P_ = 5; __VA_ARGS__; } break;                 \
        case 6: { constexpr int P_ = 6; __VA_ARGS__; } break;                 \
        case 7: { constexpr int P_ = 7; __VA_ARGS__; } break;                 \
        case 8: { constexpr int P_ = 8; __VA_ARGS__; } break;                 \
        default: return cudaErrorInvalidValue;                         \
    }

// blocks of the CG kernels (their partial sums go to d_gpart)
static int cg_blocks(const lrccs_ctx *c) { return std::min(c->nsm, (c->n + CG_THREADS - 1) / CG_THREADS); }

cudaError_t launch_cg_init(lrccs_ctx *c, double *cg) {
    prof_begin(c, KID_CG_INIT);
    // 8 warps a block, one pixel each: four blocks per multiprocessor
    k_cg_init<<<4 * c->nsm < 1024 ? 4 * c->nsm : 1024, CG_THREADS, 0, c->stream>>>(
        c->d_Z, c->n, c->q, c->d_G, c->d_U, c->d_Uprev, c->d_B, cg, (double *)c->d_gpart, c->d_counters + CNT_CG);
    prof_end(c, KID_CG_INIT);
    return cudaGetLastError();
}

cudaError_t launch_cg_step(lrccs_ctx *c, double *cg) {
    const int nb = cg_blocks(c);
    double *part = (double *)c->d_gpart;
    unsigned int *cnt = c->d_counters + CNT_CG;
    prof_begin(c, KID_CG_STEP);
    k_cg_dot<<<nb, CG_THREADS, 0, c->stream>>>(c->d_U, c->d_Up, c->n, cg, part, cnt);
    k_cg_update<<<nb, CG_THREADS, 0, c->stream>>>(c->d_U, c->d_Up, c->d_Uprev, c->d_G, c->n, cg, part, cnt);
    k_cg_dir<<<nb, CG_THREADS, 0, c->stream>>>(c->d_U, c->d_G, c->n, cg);
    prof_end(c, KID_CG_STEP);
    return cudaGetLastError();
}

cudaError_t launch_mean_resid(lrccs_ctx *c, const float2 *d_y, float2 *d_ytil, int nl_max) {
    if (nl_max < 1) return cudaSuccess;
    const float sx = (float)(1.0 / sqrt((double)c->nx));
    const dim3 grid((unsigned)((c->nc * nl_max + 7) / 8), (unsigned)c->q);
    DISPATCH_P(c->px, {
        prof_begin(c, KID_MEAN_RESID);
        k_mean_resid<P_><<<grid, 256, 0, c->stream>>>(d_y, c->d_T, c->d_framerows, c->d_lineptr, d_ytil, c->ny,
                                                      c->nc, c->d_twx, sx);
        prof_end(c, KID_MEAN_RESID);
    });
    return cudaGetLastError();
}
