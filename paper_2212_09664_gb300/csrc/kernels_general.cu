// kernels_general.cu -- altGDmin (Alg. 2) with general 2D sampling masks on
// sm_103a: masks whose rows are only partly sampled, such as the pseudo-radial
// golden-angle trajectories gridded onto the Cartesian grid (Sec. V).
//
// With such masks the x-direction transforms no longer cancel.  An iteration
// applies F = F_x F_y to the C r coil images d_j o u_l and keeps the result
// only at the union Omega_u of all frames' samples, stored row by row
// (FU[j][u][l], u = 0 .. n_u - 1 in ascending k-space index).  Linearity gives
//   G_k = (A_k U)^H (A_k U) = sum_{u in Omega_k} P_u,   P_u = sum_j FU_j[u]^H FU_j[u],
//   sum_k A_k^H (A_k U b_k - y_k) b_k^H = sum_j conj(d_j) o F^H [FU_j W] - Z B^H,
//   W_u = sum_{k: u in Omega_k} b_k b_k^H,
// so the iteration still costs C r forward and C r inverse 2D transforms.
//
// Kernels of one iteration (A, F and G are the line path's):
//   A  k_fwd_cols     : F_y(d_j o U) on the rows of Omega_u          -> T[j][ky][x][l]
//   A2 k_fwd_rows     : F_x of each such row, gather of its union points -> FU[j][u][l]
//   B  k_sample_gram  : P_u = sum_j FU_j[u]^H FU_j[u]                 -> Pu[u][pair]
//   C  k_solve_gen    : G_k = sum of P_u over the frame's samples, h_k, Cholesky -> B  (kernels_solve.cu)
//   D  k_sample_w     : FU_j[u] <- FU_j[u] W_u                        -> FU (in place)
//   E  k_adj_rows     : scatter a row's union points, F_x^H           -> T[j][ky][x][l]
//   F  k_adj_cols     : F_y^H and the conj(d_j) coil sum              -> Gk
//   G  k_gdqr         : gradient, GD step, QR                          (kernels_gd.cu)
// (the spectral initialisation takes any mask: kernels_init.cu).
#include <math.h>

#include <algorithm>

#include "common.cuh"
#include "fft.cuh"
#include "internal.h"

#define RMAXC 16
#define FULLMASK 0xffffffffu

#define DISPATCH_P(PV, ...)                                            \
    switch (PV) {                                                      \
        case 1: { constexpr int P_ = 1; __VA_ARGS__; } break;          \
        case 2: { constexpr int P_ = 2; __VA_ARGS__; } break;          \
        case 3: { constexpr int P_ = 3; __VA_ARGS__; } break;          \
        case 4: { constexpr int P_ = 4; __VA_ARGS__; } break;          \
        case 5: { constexpr int P_ = 5; __VA_ARGS__; } break;          \
        case 6: { constexpr int P_ = 6; __VA_ARGS__; } break;          \
        case 7: { constexpr int P_ = 7; __VA_ARGS__; } break;          \
        case 8: { constexpr int P_ = 8; __VA_ARGS__; } break;          \
        default: return cudaErrorInvalidValue;                         \
    }

// ---------------------------------------------------------------- compaction

// ucnt[i] = number of frames that sample k-space point i.
__global__ void k_union_count(const uint8_t *__restrict__ mask, int q, int n, int32_t *__restrict__ ucnt) {
    for (int i = blockIdx.x * blockDim.x + threadIdx.x; i < n; i += gridDim.x * blockDim.x) {
        int c = 0;
        for (int k = 0; k < q; ++k) c += mask[(size_t)k * n + i] != 0;
        ucnt[i] = c;
    }
}

// One block of 256 threads per row ky (nx <= 256): exclusive prefix counts of
// the row's union points (uloc, -1 off the union) and of their frame-list
// lengths (floc); the row totals go to urow[ky] and urow[ny + ky].
__global__ void __launch_bounds__(256) k_union_rows(const int32_t *__restrict__ ucnt, int ny, int nx,
                                                     int32_t *__restrict__ uloc, int32_t *__restrict__ floc,
                                                     int32_t *__restrict__ urow) {
    __shared__ int s_a[8], s_b[8];
    const int ky = blockIdx.x, x = threadIdx.x, lane = x & 31, w = x >> 5;
    const int c = x < nx ? ucnt[ky * nx + x] : 0;
    const int f = c > 0 ? 1 : 0;
    int a = f, b = c;   // inclusive warp scans
#pragma unroll
    for (int o = 1; o < 32; o <<= 1) {
        const int ta = __shfl_up_sync(FULLMASK, a, o), tb = __shfl_up_sync(FULLMASK, b, o);
        if (lane >= o) {
            a += ta;
            b += tb;
        }
    }
    if (lane == 31) {
        s_a[w] = a;
        s_b[w] = b;
    }
    __syncthreads();
    int pa = 0, pb = 0;
    for (int v = 0; v < w; ++v) {
        pa += s_a[v];
        pb += s_b[v];
    }
    if (x < nx) {
        uloc[ky * nx + x] = f ? pa + a - 1 : -1;
        floc[ky * nx + x] = pb + b - c;
    }
    if (x == (int)blockDim.x - 1) {
        urow[ky] = pa + a;
        urow[ny + ky] = pb + b;
    }
}

// Row offsets of the union points and of their frame lists: one warp, 32 rows at
// a time (ny is a multiple of 32).  One thread adding the rows one by one: 10 us;
// 4 us.
__global__ void k_union_scan(const int32_t *__restrict__ urow, int ny, int32_t *__restrict__ uptr,
                             int32_t *__restrict__ ufrow, int32_t *__restrict__ ufptr, int32_t *__restrict__ meta) {
    const int lane = threadIdx.x;
    int a = 0, b = 0;
    for (int y0 = 0; y0 < ny; y0 += 32) {
        const int ky = y0 + lane, ca = urow[ky], cb = urow[ny + ky];
        int sa = ca, sb = cb;   // inclusive warp scans
#pragma unroll
        for (int o = 1; o < 32; o <<= 1) {
            const int ta = __shfl_up_sync(FULLMASK, sa, o), tb = __shfl_up_sync(FULLMASK, sb, o);
            if (lane >= o) {
                sa += ta;
                sb += tb;
            }
        }
        uptr[ky] = a + sa - ca;
        ufrow[ky] = b + sb - cb;
        a += __shfl_sync(FULLMASK, sa, 31);
        b += __shfl_sync(FULLMASK, sb, 31);
    }
    if (lane == 0) {
        uptr[ny] = a;
        ufrow[ny] = b;
        ufptr[a] = b;
        meta[MT_NU] = a;
    }
}

// Per union point u (k-space index i): upos[i] = u, and its frames
// in ascending order at uflist[ufptr[u] ..] (a deterministic order, so that
// W_u is summed the same way on every run).
__global__ void k_union_fill(const uint8_t *__restrict__ mask, const int32_t *__restrict__ uloc,
                             const int32_t *__restrict__ floc, const int32_t *__restrict__ uptr,
                             const int32_t *__restrict__ ufrow, int q, int nx, int n, int32_t *__restrict__ upos,
                             int32_t *__restrict__ ufptr, int32_t *__restrict__ uflist) {
    for (int i = blockIdx.x * blockDim.x + threadIdx.x; i < n; i += gridDim.x * blockDim.x) {
        const int l = uloc[i];
        if (l < 0) {
            upos[i] = -1;
            continue;
        }
        const int ky = i / nx;
        const int u = uptr[ky] + l;
        upos[i] = u;
        const int f0 = ufrow[ky] + floc[i];
        ufptr[u] = f0;
        int cnt = 0;
        for (int k = 0; k < q; ++k)
            if (mask[(size_t)k * n + i]) uflist[f0 + cnt++] = k;
    }
}

// One warp per (frame k, row ky): the row's samples in ascending kx at
// idx[rowoff ..], and their union indices at fu[rowoff ..].
__global__ void k_fill_general(const uint8_t *__restrict__ mask, const int32_t *__restrict__ rowcnt,
                               const int32_t *__restrict__ rowoff, const int32_t *__restrict__ upos, int q, int ny,
                               int nx, int32_t *__restrict__ idx, int32_t *__restrict__ fu) {
    const int w = (int)((blockIdx.x * blockDim.x + threadIdx.x) >> 5), lane = threadIdx.x & 31;
    if (w >= q * ny || rowcnt[w] == 0) return;   // uniform across the warp
    const int k = w / ny, ky = w - k * ny;
    const uint8_t *m = mask + (size_t)k * ny * nx + (size_t)ky * nx;
    int pos = rowoff[w];
    for (int x0 = 0; x0 < nx; x0 += 32) {
        const int x = x0 + lane;
        const bool b = x < nx && m[x] != 0;
        const unsigned bal = __ballot_sync(FULLMASK, b);
        if (b) {
            const int p = pos + __popc(bal & ((1u << lane) - 1u));
            idx[p] = ky * nx + x;
            fu[p] = upos[ky * nx + x];
        }
        pos += __popc(bal);
    }
}

cudaError_t launch_compact_general(lrccs_ctx *c, const uint8_t *d_mask) {
    const int n = c->n, q = c->q, ny = c->ny, nx = c->nx;
    const int blocks = (n + 255) / 256;
    prof_begin(c, KID_UNION);
    k_union_count<<<blocks, 256, 0, c->stream>>>(d_mask, q, n, c->d_ucnt);
    prof_end(c, KID_UNION);
    prof_begin(c, KID_UNION);
    k_union_rows<<<ny, 256, 0, c->stream>>>(c->d_ucnt, ny, nx, c->d_uloc, c->d_floc, c->d_urow);
    prof_end(c, KID_UNION);
    prof_begin(c, KID_UNION);
    k_union_scan<<<1, 32, 0, c->stream>>>(c->d_urow, ny, c->d_uptr, c->d_ufrow, c->d_ufptr, c->d_meta);
    prof_end(c, KID_UNION);
    prof_begin(c, KID_UNION);
    k_union_fill<<<blocks, 256, 0, c->stream>>>(d_mask, c->d_uloc, c->d_floc, c->d_uptr, c->d_ufrow, q, nx, n,
                                                c->d_upos, c->d_ufptr, c->d_uflist);
    prof_end(c, KID_UNION);
    prof_begin(c, KID_FILL_GEN);
    k_fill_general<<<(q * ny * 32 + 255) / 256, 256, 0, c->stream>>>(d_mask, c->d_rowcnt, c->d_rowoff, c->d_upos,
                                                                      q, ny, nx, c->d_idx, c->d_fu);
    prof_end(c, KID_FILL_GEN);
    return cudaGetLastError();
}

// ---------------------------------------------------------------- A2, E: the row passes
//
// A row (nx x r complex values of T_j[ky], l innermost) is transformed along x
// with the two register halves of fft.cuh, N = R1 R2.  Item i = g r + l of a
// coil: its length-R1 DFT takes elements x = g + R2 m, at m R2 r + i of the row,
// and its length-R2 DFT gives x = g + R1 k2, at k2 R1 r + i, so every access to
// the row is contiguous over the items whatever the rank.  The exchange tile
// holds element (k1, j2, l) at k1 S + j2 r + l; S = r modulo 16 keeps the second
// half's reads on distinct banks.  Each thread stages its own elements by
// cp.async while the previous coil's second half runs (two tiles, one block
// barrier per step) and transforms them in place.  A block takes the coils of
// its group, CB at a time (small ranks), of one row ky.
//
// Which points of the row exist: the union points (iterations), or with ftab
// only those that frame k0 + l samples (the frames' normal operators): 16-bit
// masks per (frame, row, g), over k2 for the forward pass ([..][0..15]) and over
// m for the adjoint ([..][16..31]).
struct RowArgs {
    const int32_t *usedrows, *uptr, *upos;
    const uint16_t *ftab;      // NULL: every union point
    const float2 *tw;          // [j2][k1] twiddles with the scale 1 / sqrt(nx)
    int ny, r, nc, nu, S, CB, k0, q;
};

template <int P>
struct RowPlan {
    static constexpr int NX = 32 * P, R1 = fft::Plan<NX>::R1, R2 = fft::Plan<NX>::R2, NG = R1 > R2 ? R1 : R2;
};

// the row's union index of every x (-1: none) into s_up; ends with a barrier
LRCCS_DEV void row_positions(int16_t *s_up, const RowArgs &a, int ky, int nx) {
    const int u0 = a.uptr[ky];
    for (int x = threadIdx.x; x < nx; x += blockDim.x) {
        const int u = __ldg(a.upos + (size_t)ky * nx + x);
        s_up[x] = (int16_t)(u < 0 ? -1 : u - u0);
    }
    __syncthreads();
}
// the points x = g + step i, i < cnt, of column l as a bit mask
LRCCS_DEV uint32_t row_bits(const int16_t *s_up, const RowArgs &a, int ky, int g, int l, int step, int cnt, int half) {
    if (a.ftab) return a.k0 + l < a.q ? __ldg(a.ftab + ((size_t)(a.k0 + l) * a.ny + ky) * 32 + half + g) : 0u;
    uint32_t bits = 0;
    for (int i = 0; i < cnt; ++i) bits |= (uint32_t)(s_up[g + step * i] >= 0) << i;
    return bits;
}

// Measured (kernel time, L2 warm), whole rows staged by cp.async and transformed
// with shared-memory passes -> this form: 256 x 256, C = 20, r = 12, 28.9k
// points: 56 -> 55 us (DRAM: 126 MB of T in, 126 MB of its dirty lines out);
// 224 x 224, C = 18, r = 13, 8 frames: 44 -> 32 us
template <int P>
__global__ void __launch_bounds__(256, 3) k_fwd_rows(const float2 *__restrict__ T, float2 *__restrict__ FU,
                                                     const RowArgs a) {
    using PL = RowPlan<P>;
    constexpr int NX = PL::NX, R1 = PL::R1, R2 = PL::R2, NG = PL::NG;
    extern __shared__ __align__(16) float2 smem[];
    __shared__ int16_t s_up[NX];
    const int r = a.r, IT = NG * r, tile = R1 * a.S, ky = a.usedrows[blockIdx.x];
    const int slot = threadIdx.x / IT, i = threadIdx.x - slot * IT, g = i / r, l = i - g * r;
    const bool first = slot < a.CB && g < R2, second = slot < a.CB && g < R1;
    const size_t rowlen = (size_t)NX * r;
    const int u0 = a.uptr[ky], step = gridDim.y * a.CB;
    float2 *mine = smem + slot * tile;
    auto stage = [&](int j, int s) {
        if (first && j < a.nc) {
            float2 *dst = mine + s * a.CB * tile + i;
            const float2 *src = T + ((size_t)j * a.ny + ky) * rowlen + i;
#pragma unroll
            for (int m = 0; m < R1; ++m) cp_async8(dst + m * a.S, src + m * R2 * r);
        }
        cp_async_commit();
    };
    stage(blockIdx.y * a.CB + slot, 0);
    row_positions(s_up, a, ky, NX);
    const uint32_t bits = second ? row_bits(s_up, a, ky, g, l, R1, R2, 0) : 0u;
    int s = 0;
    for (int b = blockIdx.y * a.CB; b < a.nc; b += step, s ^= 1) {
        const int j = b + slot;
        float2 *ex = mine + s * a.CB * tile;
        cp_async_wait();
        if (first && j < a.nc) {
            float2 v[R1];
#pragma unroll
            for (int m = 0; m < R1; ++m) v[m] = ex[m * a.S + i];
            fft::dft_first<R1, R2, false>(v, g, a.tw, [&](int k1, float2 w) { ex[k1 * a.S + i] = w; });
        }
        __syncthreads();
        if (b + step < a.nc) stage(j + step, s ^ 1);
        if (bits != 0 && j < a.nc) {
            float2 v[R2];
            const float2 *e = ex + g * a.S + l;
#pragma unroll
            for (int j2 = 0; j2 < R2; ++j2) v[j2] = e[j2 * r];
            fft::Dft<R2, false>::run(v);
            float2 *dst = FU + ((size_t)j * a.nu + u0) * r + l;
#pragma unroll
            for (int k2 = 0; k2 < R2; ++k2)
                if (bits >> k2 & 1) dst[s_up[g + R1 * k2] * r] = v[k2];
        }
    }
}

// The row's points scattered into a zero row, transformed back along x, the
// full row written to T_j[ky] for the column pass.  Measured as above: 87 -> 48 us;
// 65 -> 36 us.
template <int P>
__global__ void __launch_bounds__(256, 3) k_adj_rows(const float2 *__restrict__ FU, float2 *__restrict__ T,
                                                     const RowArgs a) {
    using PL = RowPlan<P>;
    constexpr int NX = PL::NX, R1 = PL::R1, R2 = PL::R2, NG = PL::NG;
    extern __shared__ __align__(16) float2 smem[];
    __shared__ int16_t s_up[NX];
    const int r = a.r, IT = NG * r, tile = R1 * a.S, ky = a.usedrows[blockIdx.x];
    const int slot = threadIdx.x / IT, i = threadIdx.x - slot * IT, g = i / r, l = i - g * r;
    const bool first = slot < a.CB && g < R2, second = slot < a.CB && g < R1;
    const size_t rowlen = (size_t)NX * r;
    const int u0 = a.uptr[ky], step = gridDim.y * a.CB;
    float2 *mine = smem + slot * tile;
    row_positions(s_up, a, ky, NX);
    const uint32_t bits = first ? row_bits(s_up, a, ky, g, l, R2, R1, 16) : 0u;
    const unsigned pt = (unsigned)(r * sizeof(float2)), piece = (unsigned)(R1 * r * sizeof(float2));
    auto stage = [&](int j, int s) {   // zeros at the points that do not exist
        if (first && j < a.nc) {
            float2 *dst = mine + s * a.CB * tile + i;
            const float2 *src = FU + ((size_t)j * a.nu + u0) * r + l;
#pragma unroll
            for (int m = 0; m < R1; ++m) {
                const uint32_t on = bits & (1u << m);
                cp_async8_or_zero(dst + m * a.S, step_by(src, pt, on ? (unsigned)s_up[g + R2 * m] : 0u), on);
            }
        }
        cp_async_commit();
    };
    stage(blockIdx.y * a.CB + slot, 0);
    int s = 0;
    for (int b = blockIdx.y * a.CB; b < a.nc; b += step, s ^= 1) {
        const int j = b + slot;
        float2 *ex = mine + s * a.CB * tile;
        cp_async_wait();
        if (first && j < a.nc) {
            float2 v[R1];
#pragma unroll
            for (int m = 0; m < R1; ++m) v[m] = ex[m * a.S + i];
            fft::dft_first<R1, R2, true>(v, g, a.tw, [&](int k1, float2 w) { ex[k1 * a.S + i] = w; });
        }
        __syncthreads();
        if (b + step < a.nc) stage(j + step, s ^ 1);
        if (second && j < a.nc) {
            float2 v[R2];
            const float2 *e = ex + g * a.S + l;
#pragma unroll
            for (int j2 = 0; j2 < R2; ++j2) v[j2] = e[j2 * r];
            fft::Dft<R2, true>::run(v);
            float2 *dst = T + ((size_t)j * a.ny + ky) * rowlen + i;
#pragma unroll
            for (int k2 = 0; k2 < R2; ++k2) *step_by(dst, piece, k2) = v[k2];
        }
    }
}

// The frames' point masks of the row passes (see RowArgs): block (row ky,
// frame k), thread t < 32.
__global__ void k_point_tables(const uint8_t *__restrict__ mask, int ny, int nx, int R1, int R2,
                               uint16_t *__restrict__ tab) {
    const int ky = blockIdx.x, k = blockIdx.y, t = threadIdx.x, g = t & 15;
    const uint8_t *m = mask + ((size_t)k * ny + ky) * nx;
    const int step = t < 16 ? R1 : R2, cnt = t < 16 ? R2 : R1;
    uint32_t bits = 0;
    if (g < step)
        for (int i = 0; i < cnt; ++i) bits |= (uint32_t)(m[g + step * i] != 0) << i;
    tab[((size_t)k * ny + ky) * 32 + t] = (uint16_t)bits;
}

// ---------------------------------------------------------------- B: per-point Gram

// Block of SU union points, thread (point, 2 x 2 tile of the upper triangle):
// the points' rows FU_j[u][:] of up to `cc` coils are staged at once and every
// thread adds its four products per coil from two 16-byte reads (even r).
// Instructions issue in 82% of the cycles: 256 x 256, C = 20, r = 12, 28.9k points:
// 35 us with one (point, pair) item and a block barrier per coil, 22 us in this
// form.
template <int R>
__global__ void __launch_bounds__(256) k_sample_gram(const float2 *__restrict__ FU, float2 *__restrict__ Pu, int nu,
                                                      int nc, int cc) {
    constexpr int np = R * (R + 1) / 2, tr = (R + 1) / 2, nt = tr * (tr + 1) / 2, SU = 256 / nt;
    extern __shared__ __align__(16) float2 smem[];   // cc x SU x R
    const int u0 = blockIdx.x * SU, cnt = min(SU, nu - u0);
    const int su = threadIdx.x / nt, w = threadIdx.x - su * nt;
    int A, Bt;
    pair_of(w, tr, A, Bt);
    const bool act = su < cnt;
    float2 acc[4];
#pragma unroll
    for (int m = 0; m < 4; ++m) acc[m] = make_float2(0.f, 0.f);
    for (int j0 = 0; j0 < nc; j0 += cc) {
        const int jn = min(cc, nc - j0);
        for (int j = 0; j < jn; ++j)
            stage_row(smem + j * SU * R, FU + ((size_t)(j0 + j) * nu + u0) * R, cnt * R, threadIdx.x, blockDim.x);
        cp_async_commit();
        cp_async_wait();
        __syncthreads();
        if (act) {
            const float2 *f = smem + su * R;
#pragma unroll 4
            for (int j = 0; j < jn; ++j, f += SU * R) {
                float2 p0, p1, q0, q1;
                if constexpr (R % 2 == 0) {
                    const float4 p = *reinterpret_cast<const float4 *>(f + 2 * A);
                    const float4 q = *reinterpret_cast<const float4 *>(f + 2 * Bt);
                    p0 = make_float2(p.x, p.y), p1 = make_float2(p.z, p.w);
                    q0 = make_float2(q.x, q.y), q1 = make_float2(q.z, q.w);
                } else {
                    p0 = f[2 * A], p1 = f[min(2 * A + 1, R - 1)];
                    q0 = f[2 * Bt], q1 = f[min(2 * Bt + 1, R - 1)];
                }
                cfmac(acc[0], p0, q0);
                cfmac(acc[1], p0, q1);
                cfmac(acc[2], p1, q0);
                cfmac(acc[3], p1, q1);
            }
        }
        __syncthreads();
    }
    if (act) {
        float2 *out = Pu + (size_t)(u0 + su) * np;
#pragma unroll
        for (int m = 0; m < 4; ++m) {
            const int x = 2 * A + (m >> 1), y = 2 * Bt + (m & 1);
            if (x < R && y < R && x <= y) out[pair_index(x, y, R)] = acc[m];
        }
    }
}

// ---------------------------------------------------------------- D: times W_u

// Block of SU = 256 / R union points, thread (point su, column wb):
// W_u[:, wb] = sum over the frames k sampling u of b_k conj(b_k[wb]) in
// registers, then for every coil FU_j[u][wb] <- sum_a FU_j[u][a] W_u[a][wb].  Up
// to `cc` coils' rows are staged at once (the copies run while W_u is formed),
// read by 16 bytes.  256 x 256, C = 20, r = 12, 28.9k points: 68 us with a
// stage, a wait and two barriers per coil; 43 us with the points' frame lists
// walked in global memory (the centre's points are in every frame's list), 41 us
// with the lists staged.
template <int R>
__global__ void __launch_bounds__(256) k_sample_w(float2 *__restrict__ FU, const float2 *__restrict__ B,
                                                   const int32_t *__restrict__ ufptr,
                                                   const int32_t *__restrict__ uflist, int nu, int nc, int q, int cc) {
    constexpr int SU = 256 / R;
    extern __shared__ __align__(16) float2 smem[];
    float2 *s_f = smem;                              // cc x SU x R
    float2 *sB = smem + (size_t)cc * SU * R;         // q x R
    uint8_t *s_list = (uint8_t *)(sB + q * R);       // the points' frame lists, at most SU x q
    const int u0 = blockIdx.x * SU, cnt = min(SU, nu - u0);
    const int su = threadIdx.x / R, wb = threadIdx.x - su * R;
    const bool act = su < SU && su < cnt;
    for (int e = threadIdx.x; e < q * R; e += blockDim.x) cp_async8(sB + e, B + e);
    cp_async_commit();
    const int l0 = ufptr[u0], ln = ufptr[u0 + cnt] - l0;
    for (int e = threadIdx.x; e < ln; e += blockDim.x) s_list[e] = (uint8_t)__ldg(uflist + l0 + e);
    float2 wcol[R];
#pragma unroll
    for (int a = 0; a < R; ++a) wcol[a] = make_float2(0.f, 0.f);
    for (int j0 = 0; j0 < nc; j0 += cc) {
        const int jn = min(cc, nc - j0);
        for (int j = 0; j < jn; ++j)
            stage_row(s_f + j * SU * R, FU + ((size_t)(j0 + j) * nu + u0) * R, cnt * R, threadIdx.x, blockDim.x);
        cp_async_commit();
        if (j0 == 0) {
            cp_async_wait_1();   // B is in
            __syncthreads();
            if (act) {
                const int f1 = ufptr[u0 + su + 1] - l0;
                for (int f = ufptr[u0 + su] - l0; f < f1; ++f) {
                    const float2 *bk = sB + s_list[f] * R;
                    const float2 bw = cconj(bk[wb]);
#pragma unroll
                    for (int a = 0; a < R; ++a) cfma(wcol[a], bk[a], bw);
                }
            }
        }
        cp_async_wait();
        __syncthreads();
        if (act) {
            const float2 *fs = s_f + su * R;
            float2 *dst = FU + ((size_t)j0 * nu + u0 + su) * R + wb;
#pragma unroll 2
            for (int j = 0; j < jn; ++j, fs += SU * R, dst += (size_t)nu * R) {
                float2 o = make_float2(0.f, 0.f);
                if constexpr (R % 2 == 0) {
#pragma unroll
                    for (int a = 0; a < R; a += 2) {
                        const float4 f = *reinterpret_cast<const float4 *>(fs + a);
                        cfma(o, make_float2(f.x, f.y), wcol[a]);
                        cfma(o, make_float2(f.z, f.w), wcol[a + 1]);
                    }
                } else {
#pragma unroll
                    for (int a = 0; a < R; ++a) cfma(o, fs[a], wcol[a]);
                }
                *dst = o;
            }
        }
        __syncthreads();
    }
}

// ---------------------------------------------------------------- mean step residual

// y~ = y - A_k zbar for general masks: FU (rank 1) holds F(d_j o zbar) at the
// union points; block (sample chunk, frame k) subtracts it from every coil's
// samples of frame k.
__global__ void k_mean_resid_gen(const float2 *__restrict__ y, const float2 *__restrict__ FU,
                                 const int32_t *__restrict__ fpk, const int32_t *__restrict__ fu, int nc, int nu,
                                 float2 *__restrict__ ytil) {
    const int k = blockIdx.y;
    const int f0 = fpk[k], m = fpk[k + 1] - f0;
    const int64_t base = (int64_t)nc * f0;
    for (int e = blockIdx.x * blockDim.x + threadIdx.x; e < nc * m; e += gridDim.x * blockDim.x) {
        const int j = e / m, s = e - j * m;
        const float2 a = y[base + e], b = FU[(size_t)j * nu + fu[f0 + s]];
        ytil[base + e] = make_float2(a.x - b.x, a.y - b.y);
    }
}

// ---------------------------------------------------------------- launchers

typedef void (*sgram_t)(const float2 *, float2 *, int, int, int);
typedef void (*sw_t)(float2 *, const float2 *, const int32_t *, const int32_t *, int, int, int, int);
#define RANK_TABLE(K) {K<1>, K<2>, K<3>, K<4>, K<5>, K<6>, K<7>, K<8>, K<9>, K<10>, K<11>, K<12>, K<13>, K<14>, K<15>, K<16>}
static const sgram_t kSampleGram[RMAXC] = RANK_TABLE(k_sample_gram);
static const sw_t kSampleW[RMAXC] = RANK_TABLE(k_sample_w);

// Shape of a row pass at rank r: coils at a time (a block of at most 256
// threads), exchange stride, block, shared memory, and the coil groups: the
// plan's, or the fewest rounds ceil(blocks / slots) (steps + 1) of a block's
// coil steps.
struct RowShape {
    int CB, S, threads, groups;
    size_t smem;
};
template <int P>
static RowShape row_shape(const lrccs_ctx *c, int r) {
    using PL = RowPlan<P>;
    RowShape h;
    const int it = PL::NG * r;
    h.CB = std::max(1, std::min(c->nc, 256 / it));
    h.S = PL::R2 * r + ((r - PL::R2 * r) % 16 + 16) % 16;
    h.threads = (h.CB * it + 31) / 32 * 32;
    h.smem = (size_t)2 * h.CB * PL::R1 * h.S * sizeof(float2);
    const int res = std::max(1, std::min(768 / h.threads, (int)(c->smem_sm / (h.smem + 2048))));
    const int slots = res * c->nsm, most = (c->nc + h.CB - 1) / h.CB;
    h.groups = 1;
    double cost = 1e30;
    for (int g = 1; g <= most; ++g) {
        const double v = (double)((c->n_used * g + slots - 1) / slots) * ((most + g - 1) / g + 1.0);
        if (v < cost) cost = v, h.groups = g;
    }
    if (c->plan.row_groups >= 1 && c->plan.row_groups <= 8 && c->plan.row_groups <= c->nc) h.groups = c->plan.row_groups;
    return h;
}
static RowArgs row_args(const lrccs_ctx *c, const RowShape &h, int r, int k0) {
    RowArgs a;
    a.usedrows = c->d_usedrows;
    a.uptr = c->d_uptr;
    a.upos = c->d_upos;
    a.ftab = k0 >= 0 ? c->d_ptab : nullptr;
    a.tw = c->d_twsx;
    a.ny = c->ny;
    a.r = r;
    a.nc = c->nc;
    a.nu = c->n_u;
    a.S = h.S;
    a.CB = h.CB;
    a.k0 = k0;
    a.q = c->q;
    return a;
}

cudaError_t launch_fwd_rows_r(lrccs_ctx *c, int r, int k0) {
    DISPATCH_P(c->px, {
        const RowShape h = row_shape<P_>(c, r);
        prof_begin(c, KID_FWD_ROWS);
        k_fwd_rows<P_><<<dim3(c->n_used, h.groups), h.threads, h.smem, c->stream>>>(c->d_T, c->d_FU,
                                                                                    row_args(c, h, r, k0));
        prof_end(c, KID_FWD_ROWS);
    });
    return cudaGetLastError();
}

cudaError_t launch_adj_rows_r(lrccs_ctx *c, int r, int k0) {
    DISPATCH_P(c->px, {
        const RowShape h = row_shape<P_>(c, r);
        prof_begin(c, KID_ADJ_ROWS);
        k_adj_rows<P_><<<dim3(c->n_used, h.groups), h.threads, h.smem, c->stream>>>(c->d_FU, c->d_T,
                                                                                    row_args(c, h, r, k0));
        prof_end(c, KID_ADJ_ROWS);
    });
    return cudaGetLastError();
}

// d_ptab <- the loaded masks' point tables (before launch_*_rows_r with k0 >= 0)
cudaError_t launch_point_tables(lrccs_ctx *c) {
    DISPATCH_P(c->px, {
        prof_begin(c, KID_MEC_MASK);
        k_point_tables<<<dim3(c->ny, c->q), 32, 0, c->stream>>>(c->d_maskc, c->ny, c->nx, RowPlan<P_>::R1,
                                                                RowPlan<P_>::R2, c->d_ptab);
        prof_end(c, KID_MEC_MASK);
    });
    return cudaGetLastError();
}

// coils staged at once by the point kernels: at most 48 KB, so that four blocks share a multiprocessor
static int point_coils(const lrccs_ctx *c, int su, int r) {
    return std::max(1, std::min(c->nc, (int)(49152 / ((size_t)su * r * sizeof(float2)))));
}

static cudaError_t launch_sample_gram(lrccs_ctx *c) {
    const int r = c->r, tr = (r + 1) / 2, su = 256 / (tr * (tr + 1) / 2), cc = point_coils(c, su, r);
    prof_begin(c, KID_SAMPLE_GRAM);
    kSampleGram[r - 1]<<<(c->n_u + su - 1) / su, 256, (size_t)cc * su * r * sizeof(float2), c->stream>>>(
        c->d_FU, c->d_Pu, c->n_u, c->nc, cc);
    prof_end(c, KID_SAMPLE_GRAM);
    return cudaGetLastError();
}

cudaError_t launch_sample_w(lrccs_ctx *c) {
    const int r = c->r, su = 256 / r, cc = point_coils(c, su, r);
    const size_t smem = ((size_t)cc * su * r + (size_t)c->q * r) * sizeof(float2) + (size_t)su * c->q;
    prof_begin(c, KID_SAMPLE_W);
    kSampleW[r - 1]<<<(c->n_u + su - 1) / su, 256, smem, c->stream>>>(c->d_FU, c->d_B, c->d_ufptr, c->d_uflist,
                                                                      c->n_u, c->nc, c->q, cc);
    prof_end(c, KID_SAMPLE_W);
    return cudaGetLastError();
}

cudaError_t launch_fwd_rows(lrccs_ctx *c) { return launch_fwd_rows_r(c, c->r, -1); }
cudaError_t launch_adj_rows(lrccs_ctx *c) { return launch_adj_rows_r(c, c->r, -1); }

cudaError_t launch_iteration_general_front(lrccs_ctx *c) {
    cudaError_t e = launch_fwd_rows(c);
    if (e != cudaSuccess) return e;
    e = launch_sample_gram(c);
    if (e != cudaSuccess) return e;
    return launch_solve(c);
}

cudaError_t launch_iteration_general_back(lrccs_ctx *c) {
    cudaError_t e = launch_sample_w(c);
    if (e != cudaSuccess) return e;
    return launch_adj_rows(c);
}

cudaError_t launch_mean_resid_general(lrccs_ctx *c, const float2 *d_y, float2 *d_ytil) {
    prof_begin(c, KID_MEAN_RESID_GEN);
    k_mean_resid_gen<<<dim3(16, c->q), 256, 0, c->stream>>>(d_y, c->d_FU, c->d_fpk, c->d_fu, c->nc, c->n_u, d_ytil);
    prof_end(c, KID_MEAN_RESID_GEN);
    return cudaGetLastError();
}

#define SET_SMEM(...) do { cudaError_t e_ = allow_smem(__VA_ARGS__, max_smem); if (e_ != cudaSuccess) return e_; } while (0)
cudaError_t configure_kernels_general(int max_smem) {
    SET_SMEM(k_fwd_rows<1>); SET_SMEM(k_fwd_rows<2>); SET_SMEM(k_fwd_rows<3>); SET_SMEM(k_fwd_rows<4>);
    SET_SMEM(k_fwd_rows<5>); SET_SMEM(k_fwd_rows<6>); SET_SMEM(k_fwd_rows<7>); SET_SMEM(k_fwd_rows<8>);
    SET_SMEM(k_adj_rows<1>); SET_SMEM(k_adj_rows<2>); SET_SMEM(k_adj_rows<3>); SET_SMEM(k_adj_rows<4>);
    SET_SMEM(k_adj_rows<5>); SET_SMEM(k_adj_rows<6>); SET_SMEM(k_adj_rows<7>); SET_SMEM(k_adj_rows<8>);
    for (int i = 0; i < RMAXC; ++i) {
        SET_SMEM(kSampleW[i]);
        SET_SMEM(kSampleGram[i]);
    }
    return cudaSuccess;
}
