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
// Sums per frame (dot products, norms) run in FP32 without error within a thread and
// in FP64 from there, in a fixed order.
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

// Per-frame sums over the pixels: thread (column l, slice) of block (b, cc)
// adds the products of f(i, l, add) over its slice of the block's pixels in FP32
// without error (fsum3: FP64 products and adds took 20.5 us of a 160 x 128 x 27 dot
// product, now 16.5; the update 18.9, now 17.7), the slices add in FP64 in a
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
    fsum3 s = {0.f, 0.f, 0.f};
    double wide = 0.0;
    if (sl < S) {
        auto add = [&](float a, float b) { fsum3_mul(s, wide, a, b); };
#pragma unroll 4
        for (int i = i0 + sl; i < i1; i += S) f(i, l, add);
    }
    s_red[threadIdx.x] = wide + fsum3_total(s);
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
        [&](int i, int l, auto add) {
            const size_t e = base + (size_t)i * w + l;
            const int k = cc * w + l;
            float2 s = make_float2(0.f, 0.f);
            if (k < q) s = csub(__ldg(Z + (size_t)i * q + k), __ldg(V + e));
            S[e] = s;
            P[e] = s;
            E[e] = make_float2(0.f, 0.f);
            add(s.x, s.x);
            add(s.y, s.y);
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
        [&](int i, int l, auto add) {
            const size_t e = base + (size_t)i * w + l;
            const float2 a = __ldg(P + e), b = __ldg(W + e);
            add(a.x, b.x);
            add(a.y, b.y);
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
        [&](int i, int l, auto add) {
            const size_t e = base + (size_t)i * w + l;
            const float2 p = __ldg(P + e), ww = __ldg(W + e);
            float2 ee = E[e], ss = S[e];
            ee.x = fmaf(a, p.x, ee.x);
            ee.y = fmaf(a, p.y, ee.y);
            ss.x = fmaf(-a, ww.x, ss.x);
            ss.y = fmaf(-a, ww.y, ss.y);
            E[e] = ee;
            S[e] = ss;
            add(ss.x, ss.x);
            add(ss.y, ss.y);
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

// ---------------------------------------------------------------- MEC-2: DFT along the frames

// Temporal transforms: every pixel's q values times the q x q DFT matrix.  A
// thread forms output f (with q even also f + q/2, whose sum differs only in the
// sign of the odd inputs, so half the products serve both) for TD_P pixels at
// once: per input frame one twiddle and four broadcast 16-byte reads feed the
// 8 complex products.  H = q/2 or q output pairs by 256 / H pixel groups fill
// the block.  192 x 192, q = 48, kernel time: 327 + 42 (the sums of its blocks) ->
// 35 us forward, 45 -> 28 us back.  The products alone would take 4.5 us at the
// FP32 rate; a third of the time is the second round of 5 blocks behind the 456
// that 77 registers a thread let run at once (192 x 160, 384 blocks: 21 and 18 us).
#define TD_P 8                  // pixels per thread
#define TD_S (TD_P + 2)         // shared stride of a frame's pixels (16-byte aligned, spread over the banks)

struct TdShape {
    int H, groups, pix;         // output pairs, pixel groups per block, pixels per block
    size_t smem;
};
__host__ __device__ inline TdShape td_shape(int q) {
    TdShape t;
    t.H = (q & 1) ? q : q / 2;
    t.groups = 256 / t.H;
    t.pix = t.groups * TD_P;
    t.smem = ((size_t)t.groups * q * TD_S + q) * sizeof(float2);
    return t;
}

// The block's sums over frames of s_g[(group q + k) TD_S + p] times tw^(f k):
// thread (group pg, f) receives its outputs f in lo (and f + H in hi, q even).
template <bool INV>
LRCCS_DEV void td_dft(const float2 *s_g, const float2 *s_tw, int q, int H, int pg, int f, float2 (&lo)[TD_P],
                      float2 (&hi)[TD_P]) {
    float2 ev[TD_P], od[TD_P];
#pragma unroll
    for (int p = 0; p < TD_P; ++p) ev[p] = od[p] = make_float2(0.f, 0.f);
    const float2 *g = s_g + (size_t)pg * q * TD_S;
    auto step = [&](float2 (&acc)[TD_P], int k, int t) {
        float2 w = s_tw[t];
        if (INV) w.y = -w.y;
        const float4 *g4 = reinterpret_cast<const float4 *>(g + k * TD_S);
#pragma unroll
        for (int p = 0; p < TD_P; p += 2) {
            const float4 v = g4[p / 2];
            cfma(acc[p], make_float2(v.x, v.y), w);
            cfma(acc[p + 1], make_float2(v.z, v.w), w);
        }
    };
    int t = 0;
    if (q & 1) {
        for (int k = 0; k < q; ++k) {
            step(ev, k, t);
            t += f;
            if (t >= q) t -= q;
        }
#pragma unroll
        for (int p = 0; p < TD_P; ++p) lo[p] = ev[p];
        return;
    }
    for (int k = 0; k < q; k += 2) {
        step(ev, k, t);
        t += f;
        if (t >= q) t -= q;
        step(od, k + 1, t);
        t += f;
        if (t >= q) t -= q;
    }
#pragma unroll
    for (int p = 0; p < TD_P; ++p) {
        lo[p] = cadd(ev[p], od[p]);
        hi[p] = csub(ev[p], od[p]);
    }
}

// Fill s_g from get(offset) at every (frame, pixel) of the block's pixels.
template <class GET>
LRCCS_DEV void td_fill(float2 *s_g, int q, int w, int n, int pix, GET get) {
    const int i0 = blockIdx.x * pix, cnt = pix * w;
    for (int cc = 0; cc * w < q; ++cc)
        for (int e = threadIdx.x; e < cnt; e += blockDim.x) {
            const int p = e / w, l = e - p * w, k = cc * w + l;
            if (k < q)
                s_g[((p / TD_P) * q + k) * TD_S + p % TD_P] =
                    i0 + p < n ? get(((size_t)cc * n + i0 + p) * w + l) : make_float2(0.f, 0.f);
        }
}

// M[:, i] = F_t (E + S0 - V)[i, :] (unitary DFT over the q frames, tw[t] =
// exp(-2 pi i t / q)); with part != NULL (the first step) also max |M| over the
// whole grid into *top.
__global__ void __launch_bounds__(256, 3) k_tdft_fwd(const float2 *__restrict__ E, const float2 *__restrict__ S0,
                                                     const float2 *__restrict__ V, const float2 *__restrict__ tw, int n,
                                                     int q, int w, float2 *__restrict__ M, double *part,
                                                     unsigned int *counter, double *top) {
    extern __shared__ __align__(16) float2 s_g[];
    const TdShape t = td_shape(q);
    float2 *s_tw = s_g + (size_t)t.groups * q * TD_S;
    __shared__ double s_r[8];
    const int i0 = blockIdx.x * t.pix, lane = threadIdx.x & 31;
    const float sc = rsqrtf((float)q);
    for (int i = threadIdx.x; i < q; i += blockDim.x) s_tw[i] = tw[i];
    td_fill(s_g, q, w, n, t.pix, [&](size_t o) {
        float2 g = cadd(E[o], S0[o]);
        if (V) g = csub(g, V[o]);
        return g;
    });
    __syncthreads();
    double mx = 0.0;   // max |M|^2
    const int pg = threadIdx.x / t.H, f0 = threadIdx.x - pg * t.H;
    if (pg < t.groups) {
        float2 lo[TD_P], hi[TD_P];
        td_dft<false>(s_g, s_tw, q, t.H, pg, f0, lo, hi);
        auto put = [&](const float2 (&v)[TD_P], int f) {
            const int cc = f / w, l = f - cc * w;
#pragma unroll
            for (int p = 0; p < TD_P; ++p) {
                const int i = i0 + pg * TD_P + p;
                if (i >= n) continue;
                const float2 m = cscale(v[p], sc);
                M[((size_t)cc * n + i) * w + l] = m;
                if (part) mx = fmax(mx, (double)m.x * m.x + (double)m.y * m.y);
            }
        };
        put(lo, f0);
        if (!(q & 1)) put(hi, f0 + t.H);
    }
    if (!part) return;
    for (int o = 16; o > 0; o >>= 1) mx = fmax(mx, __shfl_xor_sync(0xffffffffu, mx, o));
    if (lane == 0) s_r[threadIdx.x >> 5] = mx;
    __syncthreads();
    if (threadIdx.x == 0) {
        for (int x = 1; x < 8; ++x) mx = fmax(mx, s_r[x]);
        part[blockIdx.x] = mx;
    }
    if (!last_block_arrive(counter) || threadIdx.x >= 32) return;
    mx = 0.0;
    for (int b = lane; b < (int)gridDim.x; b += 32) mx = fmax(mx, __ldcg(part + b));
    for (int o = 16; o > 0; o >>= 1) mx = fmax(mx, __shfl_xor_sync(0xffffffffu, mx, o));
    if (lane == 0) *top = sqrt(mx);
}

// sum |M - Mprev|^2 and sum |Mprev|^2 over the frames k < q into out[0], out[1]
// (blocks along the pixels, chunks).  FP32 without error within a warp (fsum3; a
// difference is its rounded value d and that rounding e, exactly), FP64 from
// there, in a fixed order.  FP64 work bounds every form that does more of it
// (192 x 192, q = 48: 43 us all in FP64, 52 us with a range test and an FP64 side
// path at each product), so one test covers an entry's four values and an entry
// outside the range goes to FP64 as a whole: 21 us, and the warps add in FP32 too:
// 19 us.  As a part of k_tdft_fwd, where few warps are in flight, FP32 pairs took
// 28 us and lost the squares that leave the FP32 range.
#define TD_CHANGE_BLOCKS 1024   // at most
LRCCS_DEV void td_diff(fsum3 &s, float d, float e) {   // (d + e)^2, |e| at most half an ulp of d
    fsum3_product(s, d, d);
    const float a = 2.f * d, p = __fmul_rn(a, e);
    float f;
    two_sum(s.b, p, s.b, f);
    s.c += f + (fmaf(a, e, -p) + e * e);
}
LRCCS_DEV fsum3 td_warp_sum(fsum3 s) {   // the same in every lane
#pragma unroll
    for (int o = 16; o > 0; o >>= 1) {
        const float a = __shfl_xor_sync(0xffffffffu, s.a, o), b = __shfl_xor_sync(0xffffffffu, s.b, o);
        const float c = __shfl_xor_sync(0xffffffffu, s.c, o);
        float e, f, g;
        two_sum(s.a, a, s.a, e);
        two_sum(s.b, b, s.b, f);
        two_sum(s.b, e, s.b, g);
        s.c = (s.c + c) + (f + g);
    }
    return s;
}
__global__ void __launch_bounds__(256) k_tdft_change(const float2 *__restrict__ M, const float2 *__restrict__ Mprev,
                                                     int n, int q, int w, double *part, unsigned int *counter,
                                                     double *out) {
    __shared__ fsum3 s_f[2][8];
    __shared__ double s_w[2][8];
    const unsigned total = (unsigned)n * w;
    const int cc = blockIdx.y, live = min(w, q - cc * w), lane = threadIdx.x & 31;
    const float2 *Mc = M + (size_t)cc * total, *Pc = Mprev + (size_t)cc * total;
    double dw = 0.0, pw = 0.0;
    fsum3 dd = {0.f, 0.f, 0.f}, pp = {0.f, 0.f, 0.f};
#pragma unroll 2
    for (unsigned i = blockIdx.x * blockDim.x + threadIdx.x; i < total; i += gridDim.x * blockDim.x) {
        if (live < w && (int)(i % (unsigned)w) >= live) continue;   // columns past q
        const float2 m = __ldg(Mc + i), m0 = __ldg(Pc + i);
        float dx, ex, dy, ey;
        two_sum(m.x, -m0.x, dx, ex);
        two_sum(m.y, -m0.y, dy, ey);
        // the smallest (zeros left out) and the largest magnitude, NaN above all, as bits
        unsigned lo = ~0u, hi = 0u;
        auto span = [&](float v) {
            const unsigned b = __float_as_uint(v) & 0x7fffffffu;
            lo = min(lo, b - 1u);
            hi = max(hi, b);
        };
        span(dx);
        span(dy);
        span(m0.x);
        span(m0.y);
        if (lo >= __float_as_uint(1e-13f) && hi <= __float_as_uint(1e15f)) {
            td_diff(dd, dx, ex);
            td_diff(dd, dy, ey);
            fsum3_product(pp, m0.x, m0.x);
            fsum3_product(pp, m0.y, m0.y);
        } else {
            const double x = (double)m.x - (double)m0.x, y = (double)m.y - (double)m0.y;
            dw += x * x + y * y;
            pw += (double)m0.x * m0.x + (double)m0.y * m0.y;
        }
    }
    dd = td_warp_sum(dd);
    pp = td_warp_sum(pp);
    if (__any_sync(0xffffffffu, dw != 0.0 || pw != 0.0)) {
        dw = warp_sum_d(dw);
        pw = warp_sum_d(pw);
    }
    if (lane == 0) {
        s_f[0][threadIdx.x >> 5] = dd;
        s_f[1][threadIdx.x >> 5] = pp;
        s_w[0][threadIdx.x >> 5] = dw;
        s_w[1][threadIdx.x >> 5] = pw;
    }
    __syncthreads();
    const int id = blockIdx.y * gridDim.x + blockIdx.x, nb = gridDim.x * gridDim.y;
    if (threadIdx.x < 32) {   // lane (sum, warp)
        double v = lane < 16 ? s_w[lane >> 3][lane & 7] + fsum3_total(s_f[lane >> 3][lane & 7]) : 0.0;
        for (int o = 4; o > 0; o >>= 1) v += __shfl_xor_sync(0xffffffffu, v, o);
        if (lane == 0 || lane == 8) part[2 * id + (lane >> 3)] = v;
    }
    if (!last_block_arrive(counter) || threadIdx.x >= 64) return;
    const int c = threadIdx.x >> 5;   // a warp per sum
    double r = 0.0;
    for (int x = lane; x < nb; x += 32) r += __ldcg(part + 2 * x + c);
    r = warp_sum_d(r);
    if (lane == 0) out[c] = r;
}

// E[i, :] = F_t^{-1} SThr_omega(M[:, i]): the complex soft threshold
// m (|m| - omega) / |m| for |m| > omega, else 0, then the inverse unitary DFT.
__global__ void __launch_bounds__(256, 3) k_tdft_inv(const float2 *__restrict__ M, const float2 *__restrict__ tw, int n,
                                                     int q, int w, float omega, float2 *__restrict__ E) {
    extern __shared__ __align__(16) float2 s_g[];
    const TdShape t = td_shape(q);
    float2 *s_tw = s_g + (size_t)t.groups * q * TD_S;
    const int i0 = blockIdx.x * t.pix;
    const float sc = rsqrtf((float)q);
    for (int i = threadIdx.x; i < q; i += blockDim.x) s_tw[i] = tw[i];
    td_fill(s_g, q, w, n, t.pix, [&](size_t o) {
        const float2 m = M[o];
        const float a = sqrtf(m.x * m.x + m.y * m.y);
        return a > omega ? cscale(m, (a - omega) / a) : make_float2(0.f, 0.f);
    });
    __syncthreads();
    const int pg = threadIdx.x / t.H, f0 = threadIdx.x - pg * t.H;
    if (pg >= t.groups) return;
    float2 lo[TD_P], hi[TD_P];
    td_dft<true>(s_g, s_tw, q, t.H, pg, f0, lo, hi);
    auto put = [&](const float2 (&v)[TD_P], int k) {
        const int cc = k / w, l = k - cc * w;
#pragma unroll
        for (int p = 0; p < TD_P; ++p) {
            const int i = i0 + pg * TD_P + p;
            if (i < n) E[((size_t)cc * n + i) * w + l] = cscale(v[p], sc);
        }
    };
    put(lo, f0);
    if (!(q & 1)) put(hi, f0 + t.H);
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
    return launch_images_mec(c, KID_MEC_ELEM, zbar, E, c->mec_w, Eout, Xout);
}

// M, then out[0] = max |M| (Mprev NULL: the first step), or out[1], out[2] = the sums of k_tdft_change
cudaError_t launch_tdft_fwd(lrccs_ctx *c, const float2 *E, const float2 *S0, const float2 *V, const float2 *Mprev,
                            float2 *M, double *out) {
    const TdShape t = td_shape(c->q);
    double *part = c->d_mscal + 3 * c->q;
    unsigned int *cnt = c->d_counters + CNT_MEC;
    prof_begin(c, KID_MEC_TDFT);
    k_tdft_fwd<<<(c->n + t.pix - 1) / t.pix, 256, t.smem, c->stream>>>(E, S0, V, c->d_twq, c->n, c->q, c->mec_w, M,
                                                                       Mprev ? nullptr : part, cnt, out);
    prof_end(c, KID_MEC_TDFT);
    if (Mprev) {
        dim3 grid = mec_grid(c);
        grid.x = std::max(1u, std::min(grid.x, (unsigned)TD_CHANGE_BLOCKS / grid.y));
        prof_begin(c, KID_MEC_TDFT);
        k_tdft_change<<<grid, 256, 0, c->stream>>>(M, Mprev, c->n, c->q, c->mec_w, part, cnt, out + 1);
        prof_end(c, KID_MEC_TDFT);
    }
    return cudaGetLastError();
}

cudaError_t launch_tdft_inv(lrccs_ctx *c, const float2 *M, float omega, float2 *E) {
    const TdShape t = td_shape(c->q);
    prof_begin(c, KID_MEC_TDFT);
    k_tdft_inv<<<(c->n + t.pix - 1) / t.pix, 256, t.smem, c->stream>>>(M, c->d_twq, c->n, c->q, c->mec_w, omega, E);
    prof_end(c, KID_MEC_TDFT);
    return cudaGetLastError();
}

// Scratch of the reductions: 3 q FP64 scalars, then the partials of the frame
// sums (G per column), of the temporal transform (1 per block) or of its change
// (2 per block).
size_t mec_scal_count(int n, int q, int w) {
    const int nch = (q + w - 1) / w, pix = td_shape(q).pix;
    const size_t a = (size_t)MEC_G * nch * w, b = (n + pix - 1) / pix;
    return (size_t)3 * q + std::max({a, b, (size_t)2 * TD_CHANGE_BLOCKS}) + 8;
}

cudaError_t configure_kernels_mec(int max_smem) {
    cudaError_t e = allow_smem(k_tdft_fwd, max_smem);
    return e == cudaSuccess ? allow_smem(k_tdft_inv, max_smem) : e;
}
