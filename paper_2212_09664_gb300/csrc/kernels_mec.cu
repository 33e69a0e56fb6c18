// kernels_mec.cu -- model-error correction (Alg. 3) and the per-frame normal
// operator it needs, on sm_103a.
//
// After Alg. 2, the residual measurements ytt_k = y~_k - A_k x_k (x_k = U b_k)
// still hold what the low-rank model misses.  Alg. 3 estimates it as
//   MEC-1: e_k from a few CGLS iterations on min_e ||ytt_k - A_k e||^2, per frame;
//   MEC-2: ISTA on min_E sum_k ||ytt_k - A_k e_k||^2 + omega ||F_t E||_1 with F_t
//          the DFT along the frames (a temporally sparse residual).
// Both only need the frames' normal operators N_k = A_k^H A_k and
// s_k = A_k^H ytt_k = Z[:, k] - N_k x_k (Z = [A_k^H y~_k] from the init).
//
// Frames are processed in chunks of w <= 16 columns (lrccs_mec1 chooses w),
// vectors laid out as V[c][i][l] (frame k = c w + l, pixel i), so that the
// iteration's column transforms apply N to a whole chunk at once:
//   N_k v = sum_j conj(d_j) o F^H [M_k o F(d_j o v)],
// with the per-frame sampling M_k applied between the forward and inverse
// transforms (the column passes' row tables for line masks, the row passes'
// point tables for general ones).
// Reductions per frame (dot products, norms) are FP64 in a fixed order.
#include <math.h>

#include <algorithm>

#include "common.cuh"
#include "internal.h"

#define MEC_G 152   // pixel blocks of the reduction kernels (one wave on 152 SMs)

// ---------------------------------------------------------------- per-frame sampling between the transforms

// dst (n x w) <- [N_{k0+l} src[:, l]]_l for one chunk of frames.  Column l of the
// transforms only stores and reads what frame k0 + l samples (rows, for line
// masks; points of the row passes, for general ones; nothing for frames past
// q), which is the mask.
cudaError_t launch_frame_normal_op(lrccs_ctx *c, const float2 *src, float2 *dst, int w, int k0) {
    const int e0 = c->general ? 0 : 1 + k0, es = c->general ? 0 : 1;
    cudaError_t e = launch_fwd_cols_on(c, src, w, e0, es);
    if (e == cudaSuccess && c->general) e = launch_fwd_rows_r(c, w, k0);
    if (e == cudaSuccess && c->general) e = launch_adj_rows_r(c, w, k0);
    return e == cudaSuccess ? launch_adj_cols_to(c, dst, w, e0, es) : e;
}

// ---------------------------------------------------------------- elementwise and reductions

// Element (pixel i, column l) of chunk cc is at (cc n + i) w + l; the grids are
// (pixel blocks, chunks), so an index needs one 32-bit division at most.

// X[c][i][l] = U_{t-1}[i, :] b_k (k = c w + l < q, else 0); with zbar != NULL
// (and Uprev == NULL) X[c][i][l] = zbar[i] for every frame instead.
__global__ void __launch_bounds__(256) k_mec_x(const float2 *__restrict__ Uprev, const float2 *__restrict__ B,
                                               const float2 *__restrict__ zbar, int n, int q, int r, int w,
                                               float2 *__restrict__ X) {
    const unsigned total = (unsigned)n * w;
    const int cc = blockIdx.y;
    float2 *Xc = X + (size_t)cc * total;
    for (unsigned e = blockIdx.x * blockDim.x + threadIdx.x; e < total; e += gridDim.x * blockDim.x) {
        const unsigned i = e / (unsigned)w;
        const int k = cc * w + (int)(e - i * w);
        float2 v = make_float2(0.f, 0.f);
        if (k < q) {
            if (Uprev) {
                for (int a = 0; a < r; ++a) cfma(v, __ldg(Uprev + (size_t)i * r + a), __ldg(B + (size_t)k * r + a));
            } else {
                v = __ldg(zbar + i);
            }
        }
        Xc[e] = v;
    }
}

// Z[i][k] -= V[c][i][l] (the mean's normal-operator image, online tracking).
__global__ void __launch_bounds__(256) k_mec_subz(float2 *__restrict__ Z, const float2 *__restrict__ V, int n, int q,
                                                  int w) {
    const unsigned total = (unsigned)n * w;
    const int cc = blockIdx.y;
    const float2 *Vc = V + (size_t)cc * total;
    for (unsigned e = blockIdx.x * blockDim.x + threadIdx.x; e < total; e += gridDim.x * blockDim.x) {
        const unsigned i = e / (unsigned)w;
        const int k = cc * w + (int)(e - i * w);
        if (k < q) {
            float2 *z = Z + (size_t)i * q + k;
            *z = csub(*z, __ldg(Vc + e));
        }
    }
}

// Per-frame FP64 sums over the pixels: thread (column l, slice) of block
// (b, cc) adds f(i, l) over its slice of the block's pixels, the slices add in a
// fixed tree, and the last block to arrive adds the blocks' partials (a warp per
// frame: lane-strided, then a fixed shuffle tree) and hands each frame's total
// to done(k, total).  The separate one-block finish kernel this replaces took
// 10-12 us a launch, and the indices of the pixel loop another 20 (160 x 128,
// 27 frames: dot product 27 + 11 -> 20 us; one 128 x 128 frame: 6 + 10 -> 7 us).
template <class F, class DONE>
__device__ void mec_frame_sums(int n, int w, int q, double *part, unsigned int *counter, F f, DONE done) {
    __shared__ double s_red[256];
    const int b = blockIdx.x, cc = blockIdx.y, G = gridDim.x, NW = gridDim.y * w;
    const int per = (n + G - 1) / G;
    const int i0 = min(n, b * per), i1 = min(n, i0 + per);
    const int S = blockDim.x / w, sl = threadIdx.x / w, l = threadIdx.x - sl * w;
    double acc = 0.0;
    if (sl < S) {
#pragma unroll 4
        for (int i = i0 + sl; i < i1; i += S) acc += f(i, l);
    }
    s_red[threadIdx.x] = acc;
    int h = 1;
    while (2 * h < S) h <<= 1;
    for (; h > 0; h >>= 1) {   // slices sl and sl + h, a fixed tree
        __syncthreads();
        if (sl < h && sl + h < S) s_red[threadIdx.x] += s_red[threadIdx.x + h * w];
    }
    if (threadIdx.x < w) part[(size_t)b * NW + cc * w + threadIdx.x] = s_red[threadIdx.x];
    if (!last_block_arrive(counter)) return;
    const int lane = threadIdx.x & 31;
    for (int k = threadIdx.x >> 5; k < q; k += blockDim.x >> 5) {
        double t = 0.0;
        for (int g = lane; g < G; g += 32) t += __ldcg(part + (size_t)g * NW + k);
        t = warp_sum_d(t);
        if (lane == 0) done(k, t);
    }
}

// S = Z - V, P = S, E = 0 and gamma_k = ||S_k||^2.
__global__ void __launch_bounds__(256) k_mec_start(const float2 *__restrict__ Z, const float2 *__restrict__ V, int n,
                                                   int q, int w, float2 *__restrict__ S, float2 *__restrict__ P,
                                                   float2 *__restrict__ E, double *part, unsigned int *counter,
                                                   double *gamma) {
    const int cc = blockIdx.y;
    const size_t base = (size_t)cc * n * w;
    mec_frame_sums(
        n, w, q, part, counter,
        [&](int i, int l) {
            const size_t e = base + (size_t)i * w + l;
            const int k = cc * w + l;
            float2 s = make_float2(0.f, 0.f);
            if (k < q) s = csub(__ldg(Z + (size_t)i * q + k), __ldg(V + e));
            S[e] = s;
            P[e] = s;
            E[e] = make_float2(0.f, 0.f);
            return (double)s.x * s.x + (double)s.y * s.y;
        },
        [&](int k, double t) { gamma[k] = t; });
}

// alpha_k = gamma_k / Re<p_k, w_k> (= ||A_k p_k||^2; 0 if the frame's direction has no energy)
__global__ void __launch_bounds__(256) k_mec_dot(const float2 *__restrict__ P, const float2 *__restrict__ W, int n,
                                                 int q, int w, double *part, unsigned int *counter,
                                                 const double *__restrict__ gamma, double *alpha) {
    const size_t base = (size_t)blockIdx.y * n * w;
    mec_frame_sums(
        n, w, q, part, counter,
        [&](int i, int l) {
            const size_t e = base + (size_t)i * w + l;
            const float2 a = __ldg(P + e), b = __ldg(W + e);
            return (double)a.x * b.x + (double)a.y * b.y;
        },
        [&](int k, double t) { alpha[k] = (t > 0.0 && gamma[k] > 0.0) ? gamma[k] / t : 0.0; });
}

// e += alpha p, s -= alpha w; beta_k = (new ||s_k||^2) / gamma_k, gamma_k = the new norm
__global__ void __launch_bounds__(256) k_mec_update(const float2 *__restrict__ P, const float2 *__restrict__ W,
                                                    float2 *__restrict__ E, float2 *__restrict__ S,
                                                    const double *__restrict__ alpha, int n, int q, int w, double *part,
                                                    unsigned int *counter, double *gamma, double *beta) {
    const int cc = blockIdx.y, l0 = threadIdx.x % w;
    const size_t base = (size_t)cc * n * w;
    const float a = cc * w + l0 < q ? (float)alpha[cc * w + l0] : 0.f;
    mec_frame_sums(
        n, w, q, part, counter,
        [&](int i, int l) {
            const size_t e = base + (size_t)i * w + l;
            const float2 p = __ldg(P + e), ww = __ldg(W + e);
            float2 ee = E[e], ss = S[e];
            ee.x = fmaf(a, p.x, ee.x);
            ee.y = fmaf(a, p.y, ee.y);
            ss.x = fmaf(-a, ww.x, ss.x);
            ss.y = fmaf(-a, ww.y, ss.y);
            E[e] = ee;
            S[e] = ss;
            return (double)ss.x * ss.x + (double)ss.y * ss.y;
        },
        [&](int k, double t) {
            beta[k] = gamma[k] > 0.0 ? t / gamma[k] : 0.0;
            gamma[k] = t;
        });
}

// p = s + beta p
__global__ void __launch_bounds__(256) k_mec_dir(const float2 *__restrict__ S, float2 *__restrict__ P,
                                                 const double *__restrict__ beta, int n, int q, int w) {
    const unsigned total = (unsigned)n * w;
    const int cc = blockIdx.y;
    const size_t base = (size_t)cc * total;
    for (unsigned e = blockIdx.x * blockDim.x + threadIdx.x; e < total; e += gridDim.x * blockDim.x) {
        const int k = cc * w + (int)(e % (unsigned)w);
        const float bb = k < q ? (float)beta[k] : 0.f;
        const float2 s = __ldg(S + base + e), p = P[base + e];
        P[base + e] = make_float2(fmaf(bb, p.x, s.x), fmaf(bb, p.y, s.y));
    }
}

// Caller layouts (frame k contiguous, X[k n + i]): E_out = e_k and
// X_out = zbar + U_{t-1} b_k + e_k (zbar may be NULL).
__global__ void k_mec_out(const float2 *__restrict__ E, const float2 *__restrict__ Uprev, const float2 *__restrict__ B,
                          const float2 *__restrict__ zbar, int n, int q, int r, int w, float2 *__restrict__ Eout,
                          float2 *__restrict__ Xout) {
    const size_t total = (size_t)n * q;
    for (size_t e = (size_t)blockIdx.x * blockDim.x + threadIdx.x; e < total; e += (size_t)gridDim.x * blockDim.x) {
        const int k = (int)(e / n), i = (int)(e % n);
        const float2 ev = E[((size_t)(k / w) * n + i) * w + (k % w)];
        if (Eout) Eout[e] = ev;
        if (Xout) {
            float2 x = zbar ? zbar[i] : make_float2(0.f, 0.f);
            for (int a = 0; a < r; ++a) cfma(x, Uprev[(size_t)i * r + a], B[(size_t)k * r + a]);
            Xout[e] = cadd(x, ev);
        }
    }
}

// ---------------------------------------------------------------- MEC-2: DFT along the frames

#define TD_PIX 8   // pixels per block of the temporal transforms

// M[:, i] = F_t (E + S0 - V)[i, :] (unitary DFT over the q frames, tw[t] =
// exp(-2 pi i t / q)) for TD_PIX pixels per block, and the block's max |M|,
// sum |M - Mprev|^2 and sum |Mprev|^2 (when have_prev) into part[blk][3].
__global__ void __launch_bounds__(256) k_tdft_fwd(const float2 *__restrict__ E, const float2 *__restrict__ S0,
                                                  const float2 *__restrict__ V, const float2 *__restrict__ Mprev,
                                                  const float2 *__restrict__ tw, int n, int q, int w, int have_v,
                                                  int have_prev, float2 *__restrict__ M, double *part) {
    extern __shared__ float2 s_g[];           // TD_PIX * q, then tw (q)
    float2 *s_tw = s_g + TD_PIX * q;
    __shared__ double s_r[3][256];
    const int i0 = blockIdx.x * TD_PIX;
    const float sc = rsqrtf((float)q);
    for (int t = threadIdx.x; t < q; t += blockDim.x) s_tw[t] = tw[t];
    for (int e = threadIdx.x; e < TD_PIX * q; e += blockDim.x) {
        const int p = e / q, k = e - p * q, i = i0 + p;
        float2 g = make_float2(0.f, 0.f);
        if (i < n) {
            const size_t o = ((size_t)(k / w) * n + i) * w + (k % w);
            g = cadd(E[o], S0[o]);
            if (have_v) g = csub(g, V[o]);
        }
        s_g[e] = g;
    }
    __syncthreads();
    double mx = 0.0, dd = 0.0, pp = 0.0;
    for (int e = threadIdx.x; e < TD_PIX * q; e += blockDim.x) {
        const int p = e / q, f = e - p * q, i = i0 + p;
        if (i >= n) continue;
        float2 acc = make_float2(0.f, 0.f);
        int t = 0;
        for (int k = 0; k < q; ++k) {
            cfma(acc, s_g[p * q + k], s_tw[t]);
            t += f;
            if (t >= q) t -= q;
        }
        acc = cscale(acc, sc);
        const size_t o = ((size_t)(f / w) * n + i) * w + (f % w);
        M[o] = acc;
        mx = fmax(mx, sqrt((double)acc.x * acc.x + (double)acc.y * acc.y));
        if (have_prev) {
            const float2 m0 = Mprev[o];
            const double dx = (double)acc.x - m0.x, dy = (double)acc.y - m0.y;
            dd += dx * dx + dy * dy;
            pp += (double)m0.x * m0.x + (double)m0.y * m0.y;
        }
    }
    s_r[0][threadIdx.x] = mx;
    s_r[1][threadIdx.x] = dd;
    s_r[2][threadIdx.x] = pp;
    __syncthreads();
    if (threadIdx.x == 0) {
        double a = 0.0, b = 0.0, cc = 0.0;
        for (int t = 0; t < (int)blockDim.x; ++t) {
            a = fmax(a, s_r[0][t]);
            b += s_r[1][t];
            cc += s_r[2][t];
        }
        part[(size_t)blockIdx.x * 3 + 0] = a;
        part[(size_t)blockIdx.x * 3 + 1] = b;
        part[(size_t)blockIdx.x * 3 + 2] = cc;
    }
}

// out[0] = max, out[1], out[2] = sums of the nb block partials (fixed order).
__global__ void k_tdft_finish(const double *__restrict__ part, int nb, double *out) {
    __shared__ double s_r[3][256];
    double a = 0.0, b = 0.0, c = 0.0;
    for (int t = threadIdx.x; t < nb; t += blockDim.x) {
        a = fmax(a, part[(size_t)t * 3]);
        b += part[(size_t)t * 3 + 1];
        c += part[(size_t)t * 3 + 2];
    }
    s_r[0][threadIdx.x] = a;
    s_r[1][threadIdx.x] = b;
    s_r[2][threadIdx.x] = c;
    __syncthreads();
    if (threadIdx.x == 0) {   // thread 0's own partials are in a, b, c already
        for (int t = 1; t < (int)blockDim.x; ++t) {
            a = fmax(a, s_r[0][t]);
            b += s_r[1][t];
            c += s_r[2][t];
        }
        out[0] = a;
        out[1] = b;
        out[2] = c;
    }
}

// E[i, :] = F_t^{-1} SThr_omega(M[:, i]): the complex soft threshold
// m (|m| - omega) / |m| for |m| > omega, else 0, then the inverse unitary DFT.
__global__ void __launch_bounds__(256) k_tdft_inv(const float2 *__restrict__ M, const float2 *__restrict__ tw, int n,
                                                  int q, int w, float omega, float2 *__restrict__ E) {
    extern __shared__ float2 s_g[];
    float2 *s_tw = s_g + TD_PIX * q;
    const int i0 = blockIdx.x * TD_PIX;
    const float sc = rsqrtf((float)q);
    for (int t = threadIdx.x; t < q; t += blockDim.x) s_tw[t] = tw[t];
    for (int e = threadIdx.x; e < TD_PIX * q; e += blockDim.x) {
        const int p = e / q, f = e - p * q, i = i0 + p;
        float2 m = make_float2(0.f, 0.f);
        if (i < n) {
            m = M[((size_t)(f / w) * n + i) * w + (f % w)];
            const float a = sqrtf(m.x * m.x + m.y * m.y);
            m = a > omega ? cscale(m, (a - omega) / a) : make_float2(0.f, 0.f);
        }
        s_g[e] = m;
    }
    __syncthreads();
    for (int e = threadIdx.x; e < TD_PIX * q; e += blockDim.x) {
        const int p = e / q, k = e - p * q, i = i0 + p;
        if (i >= n) continue;
        float2 acc = make_float2(0.f, 0.f);
        int t = 0;
        for (int f = 0; f < q; ++f) {
            cfma(acc, s_g[p * q + f], cconj(s_tw[t]));
            t += k;
            if (t >= q) t -= q;
        }
        E[((size_t)(k / w) * n + i) * w + (k % w)] = cscale(acc, sc);
    }
}

// ---------------------------------------------------------------- launchers

static int mec_blocks(int n) { return n < MEC_G * 64 ? (n + 63) / 64 : MEC_G; }

// blocks along the pixels of the elementwise kernels: four per multiprocessor over all chunks
static dim3 mec_grid(const lrccs_ctx *c) {
    const int need = (int)(((size_t)c->n * c->mec_w + 255) / 256);
    return dim3(std::min(need, std::max(1, 4 * c->nsm / c->mec_nch)), c->mec_nch);
}

cudaError_t launch_mec_x(lrccs_ctx *c, const float2 *Uprev, const float2 *zbar, float2 *X) {
    prof_begin(c, KID_MEC_ELEM);
    k_mec_x<<<mec_grid(c), 256, 0, c->stream>>>(Uprev, c->d_B, zbar, c->n, c->q, c->r, c->mec_w, X);
    prof_end(c, KID_MEC_ELEM);
    return cudaGetLastError();
}

cudaError_t launch_mec_subz(lrccs_ctx *c, const float2 *V) {
    prof_begin(c, KID_MEC_ELEM);
    k_mec_subz<<<mec_grid(c), 256, 0, c->stream>>>(c->d_Z, V, c->n, c->q, c->mec_w);
    prof_end(c, KID_MEC_ELEM);
    return cudaGetLastError();
}

// kind: 0 start (S = Z - V, P = S, E = 0, gamma), 1 alpha (from P, W), 2
// update (E, S, then beta and gamma), 3 direction (P = S + beta P).
cudaError_t launch_mec_cg(lrccs_ctx *c, int kind, const float2 *V) {
    const int n = c->n, q = c->q, w = c->mec_w, nch = c->mec_nch;
    double *gamma = c->d_mscal, *alpha = gamma + q, *beta = alpha + q, *part = beta + q;
    float2 *E = c->d_mec, *S = E + (size_t)nch * n * w, *P = S + (size_t)nch * n * w, *W = P + (size_t)nch * n * w;
    unsigned int *cnt = c->d_counters + CNT_MEC;
    const dim3 grid(mec_blocks(n), nch);
    prof_begin(c, KID_MEC_ELEM);
    if (kind == 0) k_mec_start<<<grid, 256, 0, c->stream>>>(c->d_Z, V, n, q, w, S, P, E, part, cnt, gamma);
    else if (kind == 1) k_mec_dot<<<grid, 256, 0, c->stream>>>(P, W, n, q, w, part, cnt, gamma, alpha);
    else if (kind == 2) k_mec_update<<<grid, 256, 0, c->stream>>>(P, W, E, S, alpha, n, q, w, part, cnt, gamma, beta);
    else k_mec_dir<<<mec_grid(c), 256, 0, c->stream>>>(S, P, beta, n, q, w);
    prof_end(c, KID_MEC_ELEM);
    return cudaGetLastError();
}

cudaError_t launch_mec_out(lrccs_ctx *c, const float2 *E, const float2 *zbar, float2 *Eout, float2 *Xout) {
    prof_begin(c, KID_MEC_ELEM);
    k_mec_out<<<4 * 152, 256, 0, c->stream>>>(E, c->d_Uprev, c->d_B, zbar, c->n, c->q, c->r, c->mec_w, Eout, Xout);
    prof_end(c, KID_MEC_ELEM);
    return cudaGetLastError();
}

cudaError_t launch_tdft_fwd(lrccs_ctx *c, const float2 *E, const float2 *S0, const float2 *V, const float2 *Mprev,
                            float2 *M, double *out) {
    const int nb = (c->n + TD_PIX - 1) / TD_PIX;
    const size_t smem = (size_t)(TD_PIX + 1) * c->q * sizeof(float2);
    double *part = c->d_mscal + 3 * c->q;
    prof_begin(c, KID_MEC_TDFT);
    k_tdft_fwd<<<nb, 256, smem, c->stream>>>(E, S0, V, Mprev, c->d_twq, c->n, c->q, c->mec_w, V != nullptr,
                                             Mprev != nullptr, M, part);
    k_tdft_finish<<<1, 256, 0, c->stream>>>(part, nb, out);
    prof_end(c, KID_MEC_TDFT);
    return cudaGetLastError();
}

cudaError_t launch_tdft_inv(lrccs_ctx *c, const float2 *M, float omega, float2 *E) {
    const int nb = (c->n + TD_PIX - 1) / TD_PIX;
    const size_t smem = (size_t)(TD_PIX + 1) * c->q * sizeof(float2);
    prof_begin(c, KID_MEC_TDFT);
    k_tdft_inv<<<nb, 256, smem, c->stream>>>(M, c->d_twq, c->n, c->q, c->mec_w, omega, E);
    prof_end(c, KID_MEC_TDFT);
    return cudaGetLastError();
}

// Scratch of the reductions: 3 q FP64 scalars, then max(G q', 3 ceil(n / TD_PIX)) partials.
size_t mec_scal_count(int n, int q, int w) {
    const int nch = (q + w - 1) / w;
    const size_t a = (size_t)MEC_G * nch * w, b = (size_t)3 * ((n + TD_PIX - 1) / TD_PIX);
    return (size_t)3 * q + (a > b ? a : b) + 8;
}
