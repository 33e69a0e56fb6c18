// kernels_gd.cu -- the GD step of Alg. 2 and its QR re-orthonormalisation as
// one cooperative kernel (one block per SM, every block resident):
//
//   phase 1  grad = Gk - Z B^H  (Gk = sum_j conj(d_j) F^H K_j from the adjoint
//            transforms, Z B^H from k_zb), partial sums of grad^H grad,
//            U^H grad, U^H U
//   -------  grid reduction; every block: eta = eta_c / ||grad||_2 (t = 1),
//            G1 = (U - eta grad)^H (U - eta grad)
//                = U^H U - eta (U^H grad + grad^H U) + eta^2 grad^H grad,
//            G1 = R1^H R1 (Cholesky), R1^{-1}
//   phase 2  U_{t+1} = (U - eta grad) R1^{-1}  (the QR step of Alg. 2 as
//            Cholesky QR), and per block the partial sums of the next
//            B-step's right-hand sides h = U_{t+1}^H Z (the solve adds the
//            blocks' rows in order); the last block out forms SD(U_t, U_{t+1})
//            from U_t^H U_{t+1} = (U^H U - eta U^H grad) R1^{-1}.
//
// G1 is formed from the exact U^H U of the current (FP32) iterate, so each
// iteration removes the loss of orthogonality of the previous one; with
// ||eta grad|| <= eta_c-sized steps G1 is well conditioned and one Cholesky
// QR pass leaves U_{t+1} orthonormal to FP32 rounding.
//
// In init mode the same kernel orthonormalises the given U+ (G1 = U+^H U+)
// and forms the first right-hand sides U_0^H Z.
// A block has one part of the pixels (several where a device has few
// multiprocessors: gdqr_parts) and its rows of U and of the gradient stay in shared
// memory across the phases; its rows of Z stream in behind phase 1 (all of them when they fit,
// else through two chunk buffers).
//
// Z B^H depends only on the B-step's result, so its own kernel k_zb forms it
// while the adjoint transforms run (a parallel branch of the iteration).
//
// Partial sums are FP32 within a block and FP64 across blocks, reduced in a
// fixed order (deterministic).  The grid barriers spin on a global counter
// with an iteration limit: a barrier that gives up sets ST_TIMEOUT and the
// kernel runs to completion with that status raised.
#include <math.h>

#include <algorithm>

#include "common.cuh"
#include "internal.h"

#define RMAXC 16   // compile-time bound on the rank
#define NTG 512    // threads per block

struct GdArgs {
    const float2 *Gk;   // n x r   sum_j conj(d_j) F^H K_j (iteration mode)
    const float2 *ZB;   // n x r   Z B^H (iteration mode)
    const float2 *Z;    // n x q   A_k^H y_k, row-major (i q + k)
    float2 *hpart;      // parts x q r partial sums of h = U_{t+1}^H Z (row b: part b)
    float2 *U;          // n x r   U_t in, U_{t+1} out
    float2 *Uprev;      // n x r   receives U_t (iteration mode)
    const float2 *Up;   // n x r   U+ (init mode)
    float2 *Gr;         // n x r   receives the gradient (iteration mode)
    float2 *part;       // parts x len partial sums
    double2 *tot;       // len totals (FP64)
    double *scal;       // SC_* scalars
    unsigned int *bar;  // [0] barrier arrivals, [1] exit count
    unsigned int *status;
    int n, q, parts, per, zs, zc, nbuf, mode;   // per: pixels per part; zc: rows of a Z chunk buffer, nbuf of them
    double eta_c;
    double eta_scale0, eta_decay;   // variable step size: eta_t = eta eta_scale0 eta_decay^k
    long long *ts;             // NULL, or GD_NTS clock64() stamps per block (phase timing)
    unsigned int spin_limit;   // polls before a grid barrier gives up (2^24 normally)
    unsigned int bar_skew;     // extra arrivals a barrier waits for (0; 1 only for the timeout test)
};

// Phase timing (measurement support): thread 0 of every block stamps clock64()
// at 9 points of the kernel, and the global timer (ns) at its entry and exit,
// when a.ts is set.
#define GD_NTS 11
#define GD_TS(i)                                                                    \
    do {                                                                            \
        if (a.ts && threadIdx.x == 0) a.ts[(size_t)blockIdx.x * GD_NTS + (i)] = clock64(); \
    } while (0)
#define GD_GT(i)                                                                    \
    do {                                                                            \
        if (a.ts && threadIdx.x == 0) {                                             \
            unsigned long long g_;                                                  \
            asm volatile("mov.u64 %0, %%globaltimer;" : "=l"(g_));                  \
            a.ts[(size_t)blockIdx.x * GD_NTS + (i)] = (long long)g_;                \
        }                                                                           \
    } while (0)

// ---------------------------------------------------------------- grid-wide steps

// grid_sync (common.cuh) is the grid-wide barrier of this cooperative kernel.

// Block b reduces entries e = b, b + G, b + 2G, ... (< len) of the P partial
// rows part[g len + e], four entries at a time (128 threads each), into FP64
// totals: per thread in g order, then a fixed shuffle tree, then the warps in
// order.
static __device__ void grid_reduce(const float2 *part, int P, int len, double2 *tot) {
    __shared__ float4 s_w[NTG / 32];   // per warp: (re.hi, re.lo, im.hi, im.lo)
    const int G = gridDim.x, l128 = threadIdx.x & 127, slot = threadIdx.x >> 7;
    for (int j0 = 0; (int)blockIdx.x + G * j0 < len; j0 += NTG / 128) {
        const int e = blockIdx.x + G * (j0 + slot);
        fsum2 re = {0.f, 0.f}, im = {0.f, 0.f};
        if (e < len)
            for (int g = l128; g < P; g += 128) {
                const float2 v = __ldcg(part + (size_t)g * len + e);
                fsum_add(re, v.x);
                fsum_add(im, v.y);
            }
        re = warp_fsum2(re);
        im = warp_fsum2(im);
        if ((threadIdx.x & 31) == 0) s_w[threadIdx.x >> 5] = make_float4(re.hi, re.lo, im.hi, im.lo);
        __syncthreads();
        if (l128 == 0 && e < len) {
            float4 w = s_w[slot * 4];
            fsum2 R = {w.x, w.y}, I = {w.z, w.w};
#pragma unroll
            for (int k = 1; k < 4; ++k) {
                w = s_w[slot * 4 + k];
                R = fsum_pair(R, fsum2{w.x, w.y});
                I = fsum_pair(I, fsum2{w.z, w.w});
            }
            tot[e] = make_double2((double)R.hi + (double)R.lo, (double)I.hi + (double)I.lo);
        }
        __syncthreads();
    }
}

// ---------------------------------------------------------------- block helpers

// Copy `rows` rows of `cols` complex values (global stride ss, shared stride
// ds) with cp.async, 16 bytes per copy when everything is 16-byte aligned.
static __device__ void stage_rows(float2 *dst, int ds, const float2 *src, int ss, int rows, int cols) {
    if ((((uintptr_t)src | smem_u32(dst)) & 15) == 0 && ((ss | ds | cols) & 1) == 0) {
        const int h = cols >> 1;
        if (h <= (int)blockDim.x) {   // fixed (piece, row-step) mapping: no per-copy division
            const int c2 = threadIdx.x % h, i0 = threadIdx.x / h, step = blockDim.x / h;
            if (i0 < step)
                for (int i = i0; i < rows; i += step) cp_async16(dst + i * ds + 2 * c2, src + (size_t)i * ss + 2 * c2);
            return;
        }
        for (int e = threadIdx.x; e < rows * h; e += blockDim.x) {
            const int i = e / h, c2 = e - i * h;
            cp_async16(dst + i * ds + 2 * c2, src + (size_t)i * ss + 2 * c2);
        }
    } else {
        for (int e = threadIdx.x; e < rows * cols; e += blockDim.x) {
            const int i = e / cols, c = e - i * cols;
            cp_async8(dst + i * ds + c, src + (size_t)i * ss + c);
        }
    }
}

// Row stride (complex values) of U and the gradient in shared memory: rows 16-byte
// aligned for even R, and eight consecutive rows on distinct banks.
template <int R>
struct GdPlan {
    static constexpr int RS = R % 4 == 0 ? R + 2 : R;
    static constexpr int TR = (R + 1) / 2, TH = TR * (TR + 1) / 2, NP = R * (R + 1) / 2;
    // 2 x 2 tiles: [grad^H grad (upper) | U^H grad (all) | U^H U (upper)], init: [U+^H U+ (upper)]
    static constexpr int T_ITER = 2 * TH + TR * TR, L_ITER = 2 * NP + R * R;
};
// pixel slices per tile: the largest power of two <= 32 with tiles x slices <= NTG
__host__ __device__ constexpr int gd_slices(int tiles) {
    int s = 1;
    while (2 * s <= 32 && 2 * s * tiles <= NTG) s *= 2;
    return s;
}

// columns 2A, 2A + 1 of a row (the last one twice past R)
template <int R>
LRCCS_DEV void gd_pair(const float2 *row, int A, float2 &p0, float2 &p1) {
    if constexpr (R % 2 == 0) {
        const float4 v = *reinterpret_cast<const float4 *>(row + 2 * A);
        p0 = make_float2(v.x, v.y);
        p1 = make_float2(v.z, v.w);
    } else {
        p0 = row[2 * A];
        p1 = row[min(2 * A + 1, R - 1)];
    }
}

// The block's partial sums of the cross-Gram tiles: thread (tile, slice) adds
// pixels slice, slice + SL, ... in two FP32 chains (SL is a power of two: one
// chain a slice would be almost twice as long as NTG / tiles slices make it),
// the slices of a tile (neighbouring lanes) add by a fixed shuffle tree, and lane
// m writes entry m to part.
template <int R, bool ITER>
static __device__ void gd_grams(const float2 *s_u, const float2 *s_a, int rows, float2 *part) {
    using PL = GdPlan<R>;
    constexpr int T = ITER ? PL::T_ITER : PL::TH, SL = gd_slices(T), RS = PL::RS;
    const int tile = threadIdx.x / SL, sl = threadIdx.x % SL;
    int kind = 2, A = 0, Bt = 0;
    if (tile < T) {
        if (!ITER || tile < PL::TH) {
            kind = ITER ? 0 : 2;
            pair_of(tile, PL::TR, A, Bt);
        } else if (tile < PL::TH + PL::TR * PL::TR) {
            kind = 1;
            A = (tile - PL::TH) / PL::TR;
            Bt = (tile - PL::TH) - A * PL::TR;
        } else {
            pair_of(tile - PL::TH - PL::TR * PL::TR, PL::TR, A, Bt);
        }
    }
    const float2 *X = kind == 0 ? s_a : s_u, *Y = kind == 2 ? s_u : s_a;
    float2 acc[4], ac2[4];
#pragma unroll
    for (int m = 0; m < 4; ++m) acc[m] = ac2[m] = make_float2(0.f, 0.f);
    if (tile < T) {
        auto add = [&](float2 (&c)[4], int i) {
            float2 p0, p1, q0, q1;
            gd_pair<R>(X + i * RS, A, p0, p1);
            gd_pair<R>(Y + i * RS, Bt, q0, q1);
            cfmac(c[0], p0, q0);
            cfmac(c[1], p0, q1);
            cfmac(c[2], p1, q0);
            cfmac(c[3], p1, q1);
        };
        int i = sl;
#pragma unroll 1   // instruction fetch counts: two pairs a turn cost 0.3 us at 192 x 192, 1.5 at 256 x 256, r = 14
        for (; i + SL < rows; i += 2 * SL) {
            add(acc, i);
            add(ac2, i + SL);
        }
        if (i < rows) add(acc, i);
#pragma unroll
        for (int m = 0; m < 4; ++m) acc[m] = cadd(acc[m], ac2[m]);
    }
#pragma unroll
    for (int o = SL / 2; o > 0; o >>= 1)
#pragma unroll
        for (int m = 0; m < 4; ++m) acc[m] = cadd(acc[m], shfl_xor2(acc[m], o));
    if (tile < T) {
#pragma unroll
        for (int m = 0; m < 4; ++m) {
            const int x = 2 * A + (m >> 1), y = 2 * Bt + (m & 1);
            if (sl != m % SL || x >= R || y >= R) continue;
            if (kind == 1) part[PL::NP + x * R + y] = acc[m];
            else if (x <= y) part[(kind == 2 && ITER ? PL::NP + R * R : 0) + pair_index(x, y, R)] = acc[m];
        }
    }
}

// R1^{-1} = (L^{-1})^H of the Hermitian positive definite G1 = L L^H in sG (R
// rows of [G1 | I], 2 R wide): one entry per thread, one barrier per pivot; row
// c of the right half ends as the unit-diagonal factor's inverse, scaled by
// 1 / sqrt(pivot c).  False (the same in every thread) when a pivot is not
// positive.  With the totals' load: one warp with the rows in registers 4.2 us
// (R = 10) and 9.2 us (R = 12), most of it instruction fetch of the unrolled
// triangles; this form 2.7 and 3.1 us.
template <int R>
static __device__ bool gd_factor(float2 *sG, float2 *sR) {
    const int e = threadIdx.x, i = e / (2 * R), j = e - i * 2 * R;
    bool ok = true;
    for (int c = 0; c < R; ++c) {
        const float d = sG[c * 2 * R + c].x;
        ok = ok && d > 0.f;
        if (i > c && i < R && (j < R ? j > c : j - R <= c)) {
            const float2 f = cscale(sG[i * 2 * R + c], 1.f / d);
            sG[e] = csub(sG[e], cmul(f, sG[c * 2 * R + j]));
        }
        __syncthreads();
    }
    if (e < R * R) {
        const int a = e / R, b = e - a * R;   // Rinv[a][b] = conj(Linv[b][a])
        sR[e] = b >= a ? cscale(cconj(sG[b * 2 * R + R + a]), rsqrtf(sG[b * 2 * R + b].x)) : make_float2(0.f, 0.f);
        if (!ok) sR[e] = make_float2(a == b ? 1.f : 0.f, 0.f);
    }
    __syncthreads();
    return ok;
}

// Stage Z rows [c0, c0 + zc) of the block's pixels into buffer `buf` (one
// committed group, empty past the last row).
static __device__ void gd_stage_z(const GdArgs &a, float2 *s_z, int i0, int rows, int chunk) {
    const int c0 = chunk * a.zc, cn = min(a.zc, rows - c0);
    if (cn > 0)
        stage_rows(s_z + (size_t)(chunk % a.nbuf) * a.zc * a.zs, a.zs, a.Z + (size_t)(i0 + c0) * a.q, a.q, cn, a.q);
    cp_async_commit();
}

// Partial sums of h = U_{t+1}^H Z over the block's pixels into hrow[k R + l]:
// thread (frame pair, LC columns, pixel slice) reads its two Z values by 16
// bytes and U's row by broadcast; the slices add in order.  Few frames leave
// many slices, so the columns are split then (LC = 2 instead of R), below 15 frames.
// Kernel time, whole -> split, 128 x 128 at r = 6 and 192 x 192 at r = 16: 4 frames 27 ->
// 21 and 41 -> 32 us, 12 frames 22.6 -> 18.9 and 35.0 -> 32.8, 16 frames 20.5 -> 18.7 and
// 34.8 -> 33.6, 32 frames 20.5 -> 20.0 and 35.2 -> 36.7.
template <int R, int LC>
static __device__ __noinline__ void gd_h(const GdArgs &a, const float2 *s_a, float2 *s_z, float2 *scr, int cap, int i0, int rows,
                            float2 *hrow) {
    constexpr int RS = GdPlan<R>::RS, NC = R / LC;
    const int t = threadIdx.x, q = a.q, tq = (q + 1) >> 1, items = tq * NC, Sh = NTG / items;
    const int hs = t / items, item = t - hs * items, cgp = item / tq, kp = item - cgp * tq;
    const bool act = hs < Sh;
    float2 pv[2 * LC];
#pragma unroll
    for (int v = 0; v < 2 * LC; ++v) pv[v] = make_float2(0.f, 0.f);
    const int nch = (rows + a.zc - 1) / a.zc;
    for (int ch = 0; ch < nch; ++ch) {
        // groups committed so far: nbuf ahead of this chunk
        if (a.nbuf == 1) cp_async_wait();
        else cp_async_wait_1();
        __syncthreads();
        if (act) {
            const int c0 = ch * a.zc, cn = min(a.zc, rows - c0);
            const float2 *z = s_z + (size_t)(ch % a.nbuf) * a.zc * a.zs + 2 * kp, *u = s_a + c0 * RS + cgp * LC;
#pragma unroll(LC <= 12 ? 2 : 1)
            for (int ii = hs; ii < cn; ii += Sh) {
                const float4 zz = *(const float4 *)(z + ii * a.zs);   // Z[k], Z[k+1] (pad column when k+1 = q)
                const float2 z0 = make_float2(zz.x, zz.y), z1 = make_float2(zz.z, zz.w);
                if constexpr (LC % 2 == 0 && R % 2 == 0) {
                    const float4 *u4 = (const float4 *)(u + ii * RS);
#pragma unroll
                    for (int l2 = 0; l2 < LC / 2; ++l2) {
                        const float4 uu = u4[l2];
                        const float2 ua = make_float2(uu.x, uu.y), ub = make_float2(uu.z, uu.w);
                        cfmac(pv[2 * l2], ua, z0);
                        cfmac(pv[LC + 2 * l2], ua, z1);
                        cfmac(pv[2 * l2 + 1], ub, z0);
                        cfmac(pv[LC + 2 * l2 + 1], ub, z1);
                    }
                } else {
#pragma unroll
                    for (int l = 0; l < LC; ++l) {
                        const float2 uu = u[ii * RS + l];
                        cfmac(pv[l], uu, z0);
                        cfmac(pv[LC + l], uu, z1);
                    }
                }
            }
        }
        if (ch + a.nbuf < nch) {
            __syncthreads();   // the chunk's buffer is free
            gd_stage_z(a, s_z, i0, rows, ch + a.nbuf);
        } else if (a.nbuf > 1) {
            cp_async_commit();
        }
    }
    // slices of V values per thread at a time, through the whole dynamic shared memory
    const int V = max(2, min(2 * LC, cap / NTG));
    for (int v0 = 0; v0 < 2 * LC; v0 += V) {
        __syncthreads();
        if (act) {
#pragma unroll
            for (int v = 0; v < 2 * LC; ++v)
                if (v >= v0 && v < v0 + V) scr[(v - v0) * NTG + t] = pv[v];
        }
        __syncthreads();
        const int vn = min(V, 2 * LC - v0);
        for (int w = t; w < vn * items; w += NTG) {
            const int dv = w / items, it = w - dv * items, v = v0 + dv;
            const int k = 2 * (it % tq) + v / LC, l = (it / tq) * LC + v % LC;
            if (k < q) {
                float2 sum = make_float2(0.f, 0.f);
#pragma unroll 8
                for (int ss = 0; ss < Sh; ++ss) sum = cadd(sum, scr[dv * NTG + ss * items + it]);
                hrow[k * R + l] = sum;
            }
        }
    }
}

// ---------------------------------------------------------------- the kernel

// Latency bounds it: two grid barriers, short phases between them.  Time from
// the first block's entry to the last one's exit (graph replay), inputs staged
// three wide, tile slices added one by one, a one-warp factorisation and Z
// re-staged when a block's rows did not fit -> this form: 64 x 64, q = 32, r = 4: 15.6 ->
// 13.3 us; 128 x 128, q = 8, r = 6: 21.4 -> 13.5 us; 192 x 192, q = 48, r = 10: 24.6 -> 21.3 us;
// 256 x 256, q = 64, r = 12: 55.0 -> 42.4 us.
// MANY: several parts a block, staged in turn by each phase (a form of its own: the
// loops alone cost the usual one up to 3 us).
template <int R, bool MANY>
__global__ void __launch_bounds__(NTG, 1) k_gdqr(GdArgs a) {
    GD_GT(9);
    using PL = GdPlan<R>;
    constexpr int RS = PL::RS, np = PL::NP, rr = R * R;
    extern __shared__ __align__(16) float2 smem[];
    const int q = a.q;
    float2 *s_u = smem;                            // per * RS : U_t (iteration) or U+ (init)
    float2 *s_a = s_u + (size_t)a.per * RS;        // per * RS : grad, then U_{t+1}
    float2 *s_z = s_a + (size_t)a.per * RS;        // nbuf * zc * zs: Z (for h = U_{t+1}^H Z)
    __shared__ float2 sG[R * 2 * R];
    __shared__ float2 sR[R * R];
    __shared__ float2 s_tot[PL::L_ITER];
    __shared__ JacobiWork s_jac;
    __shared__ int s_flag;
    __shared__ float s_eta;
    const int t = threadIdx.x, G = gridDim.x;
    int part = blockIdx.x, i0 = min(a.n, part * a.per), rows = min(a.n, i0 + a.per) - i0;
    auto next = [&](int p) {   // part p, when there is one
        if (!MANY || p >= a.parts) return false;
        part = p;
        i0 = min(a.n, p * a.per);
        rows = min(a.n, i0 + a.per) - i0;
        __syncthreads();   // the last part's rows are read
        return true;
    };
    const bool iter = a.mode == 1;
    const int len1 = iter ? PL::L_ITER : np;
    // eta as it stands at launch; block 0 updates the device copy only after
    // every block has passed the first barrier (so after every block read it)
    const double eta_in = a.scal[SC_ETA];
    const bool eta_set = a.scal[SC_ETASET] != 0.0;
    const double tcnt = eta_set ? a.scal[SC_TCNT] : 0.0;   // iterations since eta was set

    // ------------------------------------------------ phase 1: gradient and Gram partial sums
    GD_TS(0);
    do {
        stage_rows(s_u, RS, (iter ? a.U : a.Up) + (size_t)i0 * R, R, rows, R);
        cp_async_commit();
        for (int b = 0; b < a.nbuf; ++b) gd_stage_z(a, s_z, i0, MANY ? 0 : rows, b);   // streams in behind phase 1
        if (iter) {   // grad = Gk - Z B^H
            const float2 *gk = a.Gk + (size_t)i0 * R, *zb = a.ZB + (size_t)i0 * R;
            float2 *gr = a.Gr + (size_t)i0 * R;
            if constexpr (R % 2 == 0) {
                constexpr int H = R / 2;
#pragma unroll 4
                for (int e = t; e < rows * H; e += NTG) {
                    const float4 x = __ldg((const float4 *)gk + e), y = __ldg((const float4 *)zb + e);
                    const float4 g = make_float4(x.x - y.x, x.y - y.y, x.z - y.z, x.w - y.w);
                    ((float4 *)gr)[e] = g;
                    const int ii = e / H;
                    *(float4 *)(s_a + ii * RS + 2 * (e - ii * H)) = g;
                }
            } else {
#pragma unroll 4
                for (int e = t; e < rows * R; e += NTG) {
                    const float2 g = csub(__ldg(gk + e), __ldg(zb + e));
                    gr[e] = g;
                    const int ii = e / R;
                    s_a[ii * RS + (e - ii * R)] = g;
                }
            }
        }
        if (a.nbuf == 1) cp_async_wait_1();
        else cp_async_wait_2();
        __syncthreads();
        GD_TS(1);
        // partial row: [grad^H grad pairs (np) | U^H grad (rr) | U^H U pairs (np)], init: [U+^H U+ pairs]
        if (iter) gd_grams<R, true>(s_u, s_a, rows, a.part + (size_t)part * len1);
        else gd_grams<R, false>(s_u, s_a, rows, a.part + (size_t)part * len1);
    } while (next(part + G));
    GD_TS(2);
    GD_TS(3);
    grid_sync(a.bar, 1, a.status, a.spin_limit, a.bar_skew, ST_TIMEOUT);
    GD_TS(4);
    grid_reduce(a.part, a.parts, len1, a.tot);
    GD_TS(5);
    grid_sync(a.bar, 2, a.status, a.spin_limit, a.bar_skew, ST_TIMEOUT);
    GD_TS(6);
    for (int e = t; e < len1; e += NTG) {
        const double2 v = __ldcg(a.tot + e);
        s_tot[e] = make_float2((float)v.x, (float)v.y);
    }
    __syncthreads();

    // ------------------------------------------------ G1 = R1^H R1 and R1^{-1} (every block)
    if (iter) {
        const float2 *A1 = s_tot, *A2 = s_tot + np, *A3 = s_tot + np + rr;
        if (t == 0) s_eta = (float)eta_in;
        if (!eta_set) {
            // ||grad||_2^2 = lambda_max(grad^H grad) (Alg. 2, t = 1), FP32 Jacobi
            for (int p = t; p < np; p += NTG) {
                int x, y;
                pair_of(p, R, x, y);
                sR[x * R + y] = A1[p];
                sR[y * R + x] = cconj(A1[p]);
            }
            __syncthreads();
            block_jacobi<false>(sR, R, R, nullptr, 0, s_jac, 30);
            if (t == 0) {
                float lmax = 0.f;
                for (int x = 0; x < R; ++x) lmax = fmaxf(lmax, sR[x * R + x].x);
                const double gn = sqrt((double)lmax);
                const double eta = gn > 0.0 ? a.eta_c / gn : 0.0;
                s_eta = (float)eta;
                if (blockIdx.x == 0) {
                    a.scal[SC_GNORM] = gn;
                    a.scal[SC_ETA] = eta;
                    a.scal[SC_ETASET] = 1.0;
                }
            }
        }
        // the step of this iteration (constant unless a schedule is set), and
        // the schedule's counter for the next one (every block has read it)
        if (t == 0) {
            if (a.eta_scale0 != 1.0 || a.eta_decay != 1.0)
                s_eta = (float)((double)s_eta * a.eta_scale0 * pow(a.eta_decay, tcnt));
            if (blockIdx.x == 0) a.scal[SC_TCNT] = tcnt + 1.0;
        }
        __syncthreads();
        const float eta = s_eta, eta2 = s_eta * s_eta;
        if (t < rr) {
            const int x = t / R, y = t - x * R;
            const int p = x <= y ? pair_index(x, y, R) : pair_index(y, x, R);
            const float sg = x <= y ? 1.f : -1.f;   // lower half: conjugate of the stored pair
            const float x2r = A2[x * R + y].x + A2[y * R + x].x;
            const float x2i = A2[x * R + y].y - A2[y * R + x].y;
            sG[x * 2 * R + y] =
                make_float2(A3[p].x - eta * x2r + eta2 * A1[p].x, sg * A3[p].y - eta * x2i + eta2 * sg * A1[p].y);
            sG[x * 2 * R + R + y] = make_float2(x == y ? 1.f : 0.f, 0.f);
        }
    } else if (t < rr) {
        const int x = t / R, y = t - x * R;
        const int p = x <= y ? pair_index(x, y, R) : pair_index(y, x, R);
        sG[x * 2 * R + y] = x <= y ? s_tot[p] : cconj(s_tot[p]);
        sG[x * 2 * R + R + y] = make_float2(x == y ? 1.f : 0.f, 0.f);
    }
    __syncthreads();
    if (!gd_factor<R>(sG, sR) && t == 0 && blockIdx.x == 0) atomicOr(a.status, (unsigned)ST_NOT_SPD_QR);
    GD_TS(7);
    const float etaf = iter ? s_eta : 0.f;

    // ------------------------------------------------ phase 2: U_{t+1} = (U - eta grad) R1^{-1}
    // a thread per pixel row, in place over the gradient: column l needs the
    // columns up to l only, so they are formed from the last one down
    next(blockIdx.x);
    do {
        if (MANY) {
            stage_rows(s_u, RS, (iter ? a.U : a.Up) + (size_t)i0 * R, R, rows, R);
            if (iter) stage_rows(s_a, RS, a.Gr + (size_t)i0 * R, R, rows, R);
            cp_async_commit();
            for (int b = 0; b < a.nbuf; ++b) gd_stage_z(a, s_z, i0, rows, b);
            if (a.nbuf == 1) cp_async_wait_1();
            else cp_async_wait_2();
            __syncthreads();
        }
        for (int i = t; i < rows; i += NTG) {
            asm volatile("" ::: "memory");   // one turn as a rule: keep R1^{-1} in shared memory
            float2 w[R];
#pragma unroll
            for (int m = 0; m < R; ++m) {
                w[m] = s_u[i * RS + m];
                if (iter) w[m] = csub(w[m], cscale(s_a[i * RS + m], etaf));
            }
#pragma unroll
            for (int l = R - 1; l >= 0; --l) {
                float2 v = make_float2(0.f, 0.f);
#pragma unroll
                for (int m = 0; m <= l; ++m) cfma(v, w[m], sR[m * R + l]);
                w[l] = v;
            }
#pragma unroll
            for (int m = 0; m < R; ++m) s_a[i * RS + m] = w[m];
        }
        __syncthreads();
        for (int e = t; e < rows * R; e += NTG) {
            const int ii = e / R, l = e - ii * R;
            a.U[(size_t)i0 * R + e] = s_a[ii * RS + l];
            if (iter) a.Uprev[(size_t)i0 * R + e] = s_u[ii * RS + l];
        }
        // the part's row of h partial sums, hpart[part][k R + l]
        float2 *hrow = a.hpart + (size_t)part * q * R;
        const int cap = max(2 * NTG, 2 * a.per * RS + a.nbuf * a.zc * a.zs);   // as launched
        constexpr int LS = R % 2 == 0 ? 2 : 1;
        if (NTG / ((q + 1) >> 1) > 64) gd_h<R, LS>(a, s_a, s_z, smem, cap, i0, rows, hrow);
        else gd_h<R, R>(a, s_a, s_z, smem, cap, i0, rows, hrow);
    } while (next(part + G));
    GD_TS(8);
    // the last block out: SD(U_t, U_{t+1})^2 = r - ||U_t^H U_{t+1}||_F^2 with
    // U_t^H U_{t+1} = (U_t^H U_t - eta U_t^H grad) R1^{-1} from the totals (no
    // second reduction; thread x R + y forms entry (x, y)), and the barrier
    // counters back to zero (every block is past its last barrier)
    __syncthreads();
    if (t == 0) {
        __threadfence();
        const unsigned int prev = atomicAdd(a.bar + 1, 1u);
        s_flag = prev == (unsigned)G - 1;
    }
    __syncthreads();
    if (!s_flag) {
        GD_GT(10);
        return;
    }
    double sq = 0.0;
    if (iter && t < rr) {
        const float2 *A2 = s_tot + np, *A3 = s_tot + np + rr;
        const int x = t / R, y = t - x * R;
        float2 mv = make_float2(0.f, 0.f);
#pragma unroll
        for (int m = 0; m < R; ++m) {
            if (m <= y) {
                const float2 uu = x <= m ? A3[pair_index(x, m, R)] : cconj(A3[pair_index(m, x, R)]);
                cfma(mv, csub(uu, cscale(A2[x * R + m], etaf)), sR[m * R + y]);
            }
        }
        sq = (double)mv.x * mv.x + (double)mv.y * mv.y;
    }
    // block sum in a fixed order: warps, then warp 0 over the warp sums
    __shared__ double s_sq[NTG / 32];
    sq = warp_sum_d(sq);
    if ((t & 31) == 0) s_sq[t >> 5] = sq;
    __syncthreads();
    if (t < 32) {
        double sum = t < NTG / 32 ? s_sq[t] : 0.0;
        sum = warp_sum_d(sum);
        if (t == 0) {
            if (iter) {
                const double sd2 = (double)R - sum;
                a.scal[SC_SD] = sqrt(sd2 > 0.0 ? sd2 : 0.0);
            }
            a.bar[0] = 0u;
            a.bar[1] = 0u;
        }
    }
    GD_GT(10);
}

// ---------------------------------------------------------------- Z contractions

// Z B^H (n x r): ZB[i][l] = sum_k Z[i][k] conj(B[k][l]), the data term of the
// gradient grad = Gk - Z B^H (Alg. 2).  Block = ZB_PIX pixels, thread = (pixel,
// half of the l range); the pixels' Z rows are staged with an odd row stride
// (conflict-free 8-byte loads across pixels), B is read by broadcast.
#define ZB_PIX 128
template <int R>
__global__ void __launch_bounds__(256) k_zb(const float2 *__restrict__ Z, const float2 *__restrict__ B, int n, int q,
                                            float2 *__restrict__ ZB) {
    extern __shared__ __align__(16) float2 smem[];
    constexpr int RH = (R + 1) / 2;
    const int zs = q | 1;
    float2 *s_z = smem;               // ZB_PIX * zs
    float2 *s_b = s_z + ZB_PIX * zs;  // q * R
    const int i0 = blockIdx.x * ZB_PIX, cn = min(ZB_PIX, n - i0);
    for (int e = threadIdx.x; e < cn * q; e += blockDim.x) {
        const int ii = e / q, k = e - ii * q;
        cp_async8(s_z + ii * zs + k, Z + (size_t)i0 * q + e);
    }
    for (int e = threadIdx.x; e < q * R; e += blockDim.x) cp_async8(s_b + e, B + e);
    cp_async_commit();
    cp_async_wait();
    __syncthreads();
    const int p = threadIdx.x & (ZB_PIX - 1), h = threadIdx.x / ZB_PIX;
    if (p >= cn) return;
    const int l0 = h * RH, nl = min(RH, R - l0);
    float2 acc[RH];
#pragma unroll
    for (int j = 0; j < RH; ++j) acc[j] = make_float2(0.f, 0.f);
    const float2 *zr = s_z + p * zs;
#pragma unroll 4
    for (int k = 0; k < q; ++k) {
        const float2 z = zr[k];
#pragma unroll
        for (int j = 0; j < RH; ++j)
            if (j < nl) cfmac(acc[j], s_b[k * R + l0 + j], z);   // conj(b) z
    }
#pragma unroll
    for (int j = 0; j < RH; ++j)
        if (j < nl) ZB[(size_t)(i0 + p) * R + l0 + j] = acc[j];
}

// ---------------------------------------------------------------- launcher

typedef void (*gd_kernel_t)(GdArgs);
#define GD_TABLE(M) {k_gdqr<1, M>,  k_gdqr<2, M>,  k_gdqr<3, M>,  k_gdqr<4, M>,  k_gdqr<5, M>,  k_gdqr<6, M>, \
                     k_gdqr<7, M>,  k_gdqr<8, M>,  k_gdqr<9, M>,  k_gdqr<10, M>, k_gdqr<11, M>, k_gdqr<12, M>, \
                     k_gdqr<13, M>, k_gdqr<14, M>, k_gdqr<15, M>, k_gdqr<16, M>}
static const gd_kernel_t kGd[2][RMAXC] = {GD_TABLE(false), GD_TABLE(true)};
static int g_gd_static_smem[2][RMAXC];
#define GD_STATIC_MAX 16384   // no rank's static shared memory is above this (14880 bytes at 16)

static cudaError_t configure_gd(int max_smem, bool many) {
    for (int i = 0; i < RMAXC; ++i) {
        cudaFuncAttributes fa;
        cudaError_t e = cudaFuncGetAttributes(&fa, kGd[many][i]);
        if (e != cudaSuccess) return e;
        if (fa.sharedSizeBytes > GD_STATIC_MAX) return cudaErrorInvalidConfiguration;
        g_gd_static_smem[many][i] = (int)fa.sharedSizeBytes;
        e = cudaFuncSetAttribute(kGd[many][i], cudaFuncAttributeMaxDynamicSharedMemorySize,
                                 max_smem - (int)fa.sharedSizeBytes);
        if (e != cudaSuccess) return e;
    }
    return cudaSuccess;
}
cudaError_t configure_kernels_gd(int max_smem) { return configure_gd(max_smem, false); }
// The form for several parts a block, loaded by the contexts that use it only: with
// its 16 kernels beside the usual ones the others' code lies elsewhere, and an
// iteration at 192 x 192, r = 10 took 2 us more.
cudaError_t configure_kernels_gd_many(int max_smem) { return configure_gd(max_smem, true); }

// Z row stride in shared memory: q rounded up to 2 mod 4 complex values, so
// that 16-byte loads of consecutive pixels' rows hit distinct banks.
static int z_stride(int q) { return ((q + 1) | 3) - 1; }

// Shared memory of k_gdqr for a part's rows of U and of the gradient.
static size_t gd_fixed(int n, int r, int parts) {
    const int per = (n + parts - 1) / parts, rs = r % 4 == 0 ? r + 2 : r;
    return (size_t)2 * per * rs * sizeof(float2);
}

// Parts the n pixels are cut into for `blocks` blocks: as many, unless their rows
// of U and the gradient (rank up to rmax) and four rows of Z leave a block's
// shared memory, which few multiprocessors cause (65536 pixels at rank 16: fewer
// than 89 of them, a partition of the device): then two or more a block.
int gdqr_parts(int n, int q, int rmax, int blocks, int smem_optin) {
    for (int m = 1;; ++m) {
        bool fits = smem_optin <= 0;   // no device to ask: sizes only
        int r = 1;
        while (!fits && r <= rmax &&
               gd_fixed(n, r, m * blocks) + 4 * z_stride(q) * sizeof(float2) + GD_STATIC_MAX <= (size_t)smem_optin)
            ++r;
        fits = fits || r > rmax;
        if (fits || m * blocks >= n) return m * blocks;
    }
}

cudaError_t launch_gdqr(lrccs_ctx *c, int mode) {
    const int r = c->r, q = c->q, G = c->gd_grid;
    if (r < 1 || r > RMAXC) return cudaErrorInvalidValue;
    const int zs = z_stride(q);
    const int per = (c->n + c->gd_parts - 1) / c->gd_parts;
    const size_t fixed = gd_fixed(c->n, r, c->gd_parts);
    const bool many = c->gd_parts > G;
    const size_t avail = (size_t)(c->dev_smem_optin - g_gd_static_smem[many][r - 1]);
    if (fixed + 4 * zs * sizeof(float2) > avail) return cudaErrorInvalidConfiguration;
    // Z in one piece, or through two buffers of as many rows as fit
    const int rows = (int)((avail - fixed) / (zs * sizeof(float2)));
    const int nbuf = rows >= per ? 1 : 2, zc = nbuf == 1 ? per : rows / 2;
    GdArgs a;
    a.Gk = c->d_Up;
    a.ZB = c->d_ZB;
    a.Z = c->d_Z;
    a.hpart = c->d_hpart;
    a.U = c->d_U;
    a.Uprev = c->d_Uprev;
    a.Up = c->d_Up;
    a.Gr = c->d_G;
    a.part = c->d_gpart;
    a.tot = c->d_tot;
    a.scal = c->d_scal;
    a.bar = c->d_counters + CNT_BAR;
    a.status = c->d_status;
    a.n = c->n;
    a.q = q;
    a.parts = c->gd_parts;
    a.per = per;
    a.zs = zs;
    a.zc = zc;
    a.nbuf = nbuf;
    a.mode = mode;
    a.eta_c = c->prm.eta_c;
    a.eta_scale0 = c->prm.eta_scale0 > 0.0 ? c->prm.eta_scale0 : 1.0;
    a.eta_decay = c->prm.eta_decay > 0.0 ? c->prm.eta_decay : 1.0;
    a.spin_limit = 1u << 24;
    a.bar_skew = 0;
    a.ts = mode == 1 ? c->d_gdts : nullptr;   // also in captured iterations (phase timing on)
    if (c->test_timeout && !c->capturing) {   // lrccs_test_wait_timeout: this launch only
        a.spin_limit = 1u << 16;
        a.bar_skew = 1;
        c->test_timeout = 0;
    }
    void *args[] = {&a};
    // the h slices go through all of it, two values per thread at least
    const size_t smem = std::max(fixed + (size_t)nbuf * zc * zs * sizeof(float2), (size_t)2 * NTG * sizeof(float2));
    prof_begin(c, KID_GDQR);
    cudaError_t e = cudaLaunchCooperativeKernel((const void *)kGd[many][r - 1], dim3(G), dim3(NTG), args, smem, c->stream);
    prof_end(c, KID_GDQR);
    return e;
}

typedef void (*zb_kernel_t)(const float2 *, const float2 *, int, int, float2 *);
#define RANK_TABLE(K) {K<1>, K<2>, K<3>, K<4>, K<5>, K<6>, K<7>, K<8>, K<9>, K<10>, K<11>, K<12>, K<13>, K<14>, K<15>, K<16>}
static const zb_kernel_t kZb[RMAXC] = RANK_TABLE(k_zb);

static size_t zb_smem(int q, int r) { return ((size_t)ZB_PIX * (q | 1) + (size_t)q * r) * sizeof(float2); }
// dst (n x r) <- Z B^H of an n x q Z and a q x r B (b_k contiguous)
void launch_zb_of(lrccs_ctx *c, const float2 *Z, const float2 *B, float2 *dst) {
    kZb[c->r - 1]<<<(c->n + ZB_PIX - 1) / ZB_PIX, 256, zb_smem(c->q, c->r), c->stream>>>(Z, B, c->n, c->q, dst);
}
// d_ZB <- Z B^H (the data term of the next gradient), from the current B.
cudaError_t launch_zb(lrccs_ctx *c) {
    if (c->r < 1 || c->r > RMAXC) return cudaErrorInvalidValue;
    prof_begin(c, KID_ZB);
    launch_zb_of(c, c->d_Z, c->d_B, c->d_ZB);
    prof_end(c, KID_ZB);
    return cudaGetLastError();
}

cudaError_t configure_kernels_zh(int max_smem) {
    for (int i = 0; i < RMAXC; ++i) {
        const int r = i + 1;
        const size_t a = zb_smem(128, r);   // the largest q
        if ((int)a > max_smem) return cudaErrorInvalidConfiguration;
        cudaError_t e = cudaFuncSetAttribute(kZb[i], cudaFuncAttributeMaxDynamicSharedMemorySize, (int)a);
        if (e != cudaSuccess) return e;
    }
    return cudaSuccess;
}
