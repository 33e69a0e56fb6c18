// kernels_iter.cu -- the transform kernels of one altGDmin iteration (Alg. 2,
// GDmin loop) on sm_103a.
//
// The iteration uses exact rearrangements of Alg. 2 (linearity only):
//   A_k U = H_k [F(d_j o U)]_j         -> the transforms of U are shared by every frame;
//   (A_k U)^H y_k = U^H Z[:, k]         -> the right-hand side never re-reads y;
//   sum_k A_k^H (A_k U b_k - y_k) b_k^H
//     = sum_j conj(d_j) o F^H [FU_j[i,:] W_i] - Z B^H,   W_i = sum_{k: i in Omega_k} b_k b_k^H.
// With masks that are unions of full k-space rows, H_k keeps whole rows and
// W_i is constant along a row ky.  F = F_y F_x with a unitary F_x, and right
// multiplication by W_ky (acting on the rank index) commutes with F_x, so
//   F_x^H [F_x(T_j[ky, :]) W_ky] = T_j[ky, :] W_ky,   T_j = F_y(d_j o U),
// and by Parseval the row Gram FU^H FU of a row equals T^H T of the same row:
// one iteration needs only the C r column transforms F_y and F_y^H.
//
// Kernels (one launch each per iteration; C is in kernels_solve.cu, I and F in kernels_gd.cu;
// when every sampled row fits one block's shared memory, k_bstep in
// kernels_solve.cu does B, C, D and I in one cooperative launch):
//   A k_fwd_cols  : F_y of d_j o U over column tiles               -> T[j][ky][x][l] (sampled rows)
//   B k_row_gram  : coil-summed row Gram sum_j T_j^H T_j per sampled row -> P[ky] (clusters)
//   C k_solve     : G_k = sum of its rows' P, h_k (sum of k_gdqr's partial rows), Cholesky -> B
//   I k_zb        : Z B^H, on a parallel branch beside D and E          -> ZB
//   D k_row_w     : T_j[ky, :] <- T_j[ky, :] W_ky                    -> T (in place)
//   E k_adj_cols  : F_y^H, conj(d_j) coil sum                      -> Gk
//   F k_gdqr      : grad = Gk - Z B^H, eta (t = 1), U - eta grad and its
//                   Cholesky QR, partial sums of the next h = U^H Z, SD (kernels_gd.cu)
// The column passes A and E load straight into registers; the row passes stage
// their rows into shared memory with cp.async.
#include <cooperative_groups.h>
#include <math.h>

#include <algorithm>

#include "common.cuh"
#include "fft.cuh"
#include "internal.h"

namespace cg = cooperative_groups;

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

#define RMAXC 16   // compile-time bound on the rank

// ---------------------------------------------------------------- A: forward, along y
//
// The transforms along y act on the flat columns c = x r + l (rows of nx r
// complex values) independently, so both column passes tile the flat columns
// in groups of COLW = 16: a row of a tile is one 128-byte line whatever the
// rank, and a half-warp holds one row (tiles of 8 columns measured 15.7 / 17.7 us
// at 192 x 192 but 56 / 68 us at 256 x 256: half-lines).  A block of 16 max(R1, R2) threads
// (N = R1 R2, fft.cuh) takes one tile through the coils of its group: thread
// (lane, group g) runs the length-R1 DFT of rows g + R2 m, the groups exchange
// through shared memory once per coil (one block barrier: two exchange tiles),
// and thread (lane, g) finishes with the length-R2 DFT of rows g + R1 k2.  The
// tiles sit in L2; instructions issue in just under half of the forward and over a
// third of the adjoint pass's cycles, the waits are for loads first (192 x 192,
// C = 12, r = 10, caches cold, 18 warps a multiprocessor).  Both cost, so every shared address is a
// constant offset from a per-thread base, the scale rides in the twiddles, and a
// half-warp stages the coil map's few x of its own rows by cp.async one coil
// ahead, which needs no further block barrier.
//
// Which rows are sampled comes as bit tables (k_structure): entry e holds, per
// group, the rows of pass 2 of the forward transform ([e][0..15]) and of pass 1
// of the adjoint ([e][16..31]); column l uses entry e0 + l estep.
#define COLW 16

template <int P>
struct ColPlan {
    static constexpr int NY = 32 * P, R1 = fft::Plan<NY>::R1, R2 = fft::Plan<NY>::R2;
    static constexpr int NG = R1 > R2 ? R1 : R2, NT = COLW * NG;
};

// x values a tile of COLW flat columns can touch at rank r
__host__ __device__ inline int col_nxt(int r) { return (COLW - 1 + r - 1) / r + 1; }

// The coil map at the rows of one group (CNT rows, rowstep apart, from src) and
// the tile's nxt x values (the nxl of them inside the image), transposed to
// dst[xi (CNT + 2) + m] (the pad keeps the 16-byte reads of different xi on
// different banks); inv = ceil(2^16 / nxt).
// Up to three x values (r >= 8) every lane's copies are worked out once.
template <int CNT>
struct MapStage {
    static constexpr int NI = (3 * CNT + COLW - 1) / COLW;
    uint32_t at[NI];   // byte offsets: source << 12 | destination, or ~0
    LRCCS_DEV void init(int rowstep, int nxt, int nxl, unsigned inv, int lane) {
#pragma unroll
        for (int i = 0; i < NI; ++i) {
            const unsigned e = lane + COLW * i, m = (e * inv) >> 16, xi = e - m * nxt;
            at[i] = ((m * rowstep + xi) << 15) | ((xi * (CNT + 2) + m) << 3);   // rows span less than 2^17 pixels
            if (e >= (unsigned)(CNT * nxt) || xi >= (unsigned)nxl) at[i] = ~0u;
        }
    }
    LRCCS_DEV void run(float2 *d, const float2 *s, int rowstep, int nxt, int nxl, unsigned inv, int lane) const {
        if (nxt <= 3) {
#pragma unroll
            for (int i = 0; i < NI; ++i)
                if (at[i] != ~0u) cp_async8((char *)d + (at[i] & 4095u), (const char *)s + (at[i] >> 12));
            return;
        }
        for (unsigned e = lane; e < (unsigned)(CNT * nxt); e += COLW) {
            const unsigned m = (e * inv) >> 16, xi = e - m * nxt;
            if (xi < (unsigned)nxl) cp_async8(d + xi * (CNT + 2) + m, s + m * rowstep + xi);
        }
    }
};

// Measured (kernel time, L2 warm), TMA-staged tiles of whole columns -> this form:
// 192 x 192, C = 12, r = 10: 17.9 -> 13.0 us; 256 x 256, C = 20, r = 12: 58 -> 41 us;
// 256 x 256, C = 32, r = 14: 136 -> 69 us.  Instructions are half of its cycles, so addresses step by
// constant multiples of one row, stores are predicated rather than branched
// round, and a tile's map copies are worked out once, not per coil (all but
// the arithmetic was half of the instructions: 15.3, 44 and 72 us before).
template <int P>
__global__ void __launch_bounds__(ColPlan<P>::NT, 768 / ColPlan<P>::NT) k_fwd_cols(
    const float2 *__restrict__ U, const float2 *__restrict__ smaps, const uint32_t *__restrict__ rowtab, int e0,
    int estep, float2 *__restrict__ T, int nx, int r, int nc, int nxt, unsigned inv, const float2 *__restrict__ g_tw) {
    using PL = ColPlan<P>;
    constexpr int NY = PL::NY, R1 = PL::R1, R2 = PL::R2, NG = PL::NG;
    extern __shared__ __align__(16) float2 smem[];   // two exchange tiles, two map stages
    const int lane = threadIdx.x & (COLW - 1), g = threadIdx.x / COLW, CG = gridDim.y;
    const int rs = nx * r, c = blockIdx.x * COLW + lane, x0 = (int)((unsigned)(blockIdx.x * COLW) / (unsigned)r);
    const int x = (int)((unsigned)c / (unsigned)r), l = c - x * r;
    const bool first = R2 == NG || g < R2;
    uint32_t rows = 0;
    if (R1 == NG || g < R1) rows = __ldg(rowtab + (e0 + l * estep) * 32 + g);
    const int mstage = nxt * (R1 + 2);
    float2 *map = smem + 2 * NY * COLW + g * mstage;
    const float2 *d = smaps + (size_t)g * nx + x0;
    const int nxl = min(nxt, nx - x0);   // x values of this tile inside the image
    MapStage<R1> ms;
    ms.init(R2 * nx, nxt, nxl, inv, lane);
    float2 u[R1];
    int j = blockIdx.y;
    d += (size_t)j * NY * nx;
    if (first) {
        ms.run(map, d, R2 * nx, nxt, nxl, inv, lane);
        cp_async_commit();
#pragma unroll
        for (int m = 0; m < R1; ++m) u[m] = __ldg(U + (size_t)(g + m * R2) * rs + c);
    }
    float2 *dst = T + ((size_t)j * NY + g) * rs + c;
    const size_t dstep = (size_t)CG * NY * rs;
    const unsigned rowbytes = (unsigned)(R1 * rs * sizeof(float2));
    float2 *ex = smem;
    for (int s = 0; j < nc; j += CG, s ^= 1) {
        if (first) {
            cp_async_wait();
            __syncwarp();
            const float4 *m4 = reinterpret_cast<const float4 *>(map + s * NG * mstage + (x - x0) * (R1 + 2));
            float2 v[R1];
#pragma unroll
            for (int m = 0; m < R1; m += 2) {
                const float4 w = m4[m / 2];
                v[m] = cmul(make_float2(w.x, w.y), u[m]);
                v[m + 1] = cmul(make_float2(w.z, w.w), u[m + 1]);
            }
            fft::dft_first<R1, R2, false>(v, g, g_tw, [&](int k1, float2 w) { ex[(k1 * R2 + g) * COLW + lane] = w; });
        }
        __syncthreads();
        d += (size_t)CG * NY * nx;
        if (first && j + CG < nc) {
            ms.run(map + (s ^ 1) * NG * mstage, d, R2 * nx, nxt, nxl, inv, lane);
            cp_async_commit();
        }
        if (rows != 0) {
            float2 v[R2];
#pragma unroll
            for (int j2 = 0; j2 < R2; ++j2) v[j2] = ex[(g * R2 + j2) * COLW + lane];
            fft::Dft<R2, false>::run(v);
#pragma unroll
            for (int k2 = 0; k2 < R2; ++k2) st_global_if(step_by(dst, rowbytes, k2), v[k2], rows & (1u << k2));
        }
        dst += dstep;
        ex = ex == smem ? smem + NY * COLW : smem;
    }
}

// ---------------------------------------------------------------- B: row Gram

// Grid (sampled rows, CG) in clusters of (1, CG): block (ky, g) stages the
// row of coils g, g + CG, ... in turn (double buffered) and accumulates
// sum_j sum_x conj(T_j[ky][x][a]) T_j[ky][x][b] (a <= b) in registers: thread =
// (2 x 2 tile of pairs, x slice).  The slices, then the CG blocks' partials
// (through distributed shared memory), are summed in a fixed order into P[ky].
template <int R>
__global__ void __launch_bounds__(256) k_row_gram(const float2 *__restrict__ T, const int32_t *__restrict__ usedrows,
                                                   float2 *__restrict__ Prow, int ny, int nx, int nc) {
    constexpr int np = R * (R + 1) / 2, tr = (R + 1) / 2, nt = tr * (tr + 1) / 2;
    constexpr int S = 256 / nt;            // x slices per tile
    extern __shared__ __align__(16) float2 smem[];
    float2 *tile0 = smem, *tile1 = smem + nx * R;
    __shared__ float2 s_red[256 * 4];
    __shared__ float2 s_part[np];
    cg::cluster_group cluster = cg::this_cluster();
    const int ky = usedrows[blockIdx.x], g = blockIdx.y, CG = gridDim.y;
    const size_t plane = (size_t)ny * nx * R;
    const float2 *row0 = T + (size_t)ky * nx * R;
    if (g < nc) stage_row(tile0, row0 + (size_t)g * plane, nx * R, threadIdx.x, blockDim.x);
    cp_async_commit();
    const int w = threadIdx.x % nt, sl = threadIdx.x / nt;
    int A, Bt;
    pair_of(w, tr, A, Bt);
    const int x0 = 2 * A, x1 = min(2 * A + 1, R - 1), y0 = 2 * Bt, y1 = min(2 * Bt + 1, R - 1);
    float2 acc[4];
#pragma unroll
    for (int m = 0; m < 4; ++m) acc[m] = make_float2(0.f, 0.f);
    int b = 0;
    for (int j = g; j < nc; j += CG, b ^= 1) {
        const float2 *tile = b ? tile1 : tile0;
        if (j + CG < nc) {
            stage_row(b ? tile0 : tile1, row0 + (size_t)(j + CG) * plane, nx * R, threadIdx.x, blockDim.x);
            cp_async_commit();
            cp_async_wait_1();
        } else {
            cp_async_wait();
        }
        __syncthreads();
        if (sl < S) {
#pragma unroll 4
            for (int x = sl; x < nx; x += S) {
                const float2 p0 = tile[x * R + x0], p1 = tile[x * R + x1];
                const float2 q0 = tile[x * R + y0], q1 = tile[x * R + y1];
                cfmac(acc[0], p0, q0);
                cfmac(acc[1], p0, q1);
                cfmac(acc[2], p1, q0);
                cfmac(acc[3], p1, q1);
            }
        }
        __syncthreads();
    }
#pragma unroll
    for (int m = 0; m < 4; ++m) s_red[m * 256 + threadIdx.x] = sl < S ? acc[m] : make_float2(0.f, 0.f);
    __syncthreads();
    for (int it = threadIdx.x; it < 4 * nt; it += blockDim.x) {
        const int m = it / nt, ww = it - m * nt;
        int a2, b2;
        pair_of(ww, tr, a2, b2);
        const int a = 2 * a2 + (m >> 1), bq = 2 * b2 + (m & 1);
        if (a < R && bq < R && a <= bq) {
            float2 sum = make_float2(0.f, 0.f);
            for (int ss = 0; ss < S; ++ss) sum = cadd(sum, s_red[m * 256 + ss * nt + ww]);
            s_part[pair_index(a, bq, R)] = sum;
        }
    }
    cluster.sync();
    if (g == 0) {
        for (int p = threadIdx.x; p < np; p += blockDim.x) {
            float2 sum = make_float2(0.f, 0.f);
            for (int k = 0; k < CG; ++k) sum = cadd(sum, cluster.map_shared_rank(s_part, k)[p]);
            Prow[(size_t)ky * np + p] = sum;
        }
    }
    cluster.sync();   // no block leaves while its partial may still be read
}

// ---------------------------------------------------------------- D: row times W

// Block (sampled row ky, coil group g): W_ky = sum over the frames k sampling
// row ky of b_k b_k^H (from B staged in shared memory), then for coils g,
// g + CG, ... in turn (double buffered) T_j[ky][x][:] <- T_j[ky][x][:] W_ky in
// place.
template <int R>
__global__ void __launch_bounds__(256) k_row_w(float2 *__restrict__ T, const float2 *__restrict__ B,
                                                const int32_t *__restrict__ usedrows,
                                                const int32_t *__restrict__ rfptr,
                                                const int32_t *__restrict__ rflist, int ny, int nx, int nc, int q) {
    extern __shared__ __align__(16) float2 smem[];
    float2 *tile0 = smem, *tile1 = smem + nx * R;
    float2 *sB = tile1 + nx * R;           // q * R
    __shared__ float2 sW[R * R];
    __shared__ int s_f[256];
    const int ky = usedrows[blockIdx.x], g = blockIdx.y, CG = gridDim.y;
    const size_t plane = (size_t)ny * nx * R;
    float2 *row0 = T + (size_t)ky * nx * R;
    for (int e = threadIdx.x; e < q * R; e += blockDim.x) cp_async8(sB + e, B + e);
    if (g < nc) stage_row(tile0, row0 + (size_t)g * plane, nx * R, threadIdx.x, blockDim.x);
    cp_async_commit();
    const int f0 = rfptr[ky], nf = rfptr[ky + 1] - f0;
    for (int f = threadIdx.x; f < nf; f += blockDim.x) s_f[f] = rflist[f0 + f];
    constexpr int NXG = 256 / R;           // x groups
    const int wb = threadIdx.x % R, xg = threadIdx.x / R;
    float2 wcol[R];
    int b = 0;
    for (int j = g; j < nc; j += CG, b ^= 1) {
        const float2 *tile = b ? tile1 : tile0;
        if (j + CG < nc) {
            stage_row(b ? tile0 : tile1, row0 + (size_t)(j + CG) * plane, nx * R, threadIdx.x, blockDim.x);
            cp_async_commit();
            cp_async_wait_1();
        } else {
            cp_async_wait();
        }
        __syncthreads();
        if (j == g) {
            for (int e = threadIdx.x; e < R * R; e += blockDim.x) {
                const int a = e / R, b = e - a * R;
                float2 acc = make_float2(0.f, 0.f);
                for (int f = 0; f < nf; ++f) cfma(acc, sB[s_f[f] * R + a], cconj(sB[s_f[f] * R + b]));
                sW[e] = acc;
            }
            __syncthreads();
#pragma unroll
            for (int a = 0; a < R; ++a) wcol[a] = sW[a * R + wb];
        }
        float2 *row = row0 + (size_t)j * plane;
        if (xg < NXG) {   // thread = (output column wb, x group): W_ky[:, wb] in registers
#pragma unroll 2
            for (int x = xg; x < nx; x += NXG) {
                const float2 *fr = tile + x * R;
                float2 o = make_float2(0.f, 0.f);
#pragma unroll
                for (int a = 0; a < R; ++a) cfma(o, fr[a], wcol[a]);
                row[x * R + wb] = o;
            }
        }
        __syncthreads();
    }
}

// ---------------------------------------------------------------- E: adjoint, along y + coil sum
// Gk = sum_j conj(d_j) o F_y^H (flat column c of coil j's row-transformed K_j);
// the - Z B^H term and the Grams are added by k_gdqr (kernels_gd.cu).
//
// Grid (flat-column tiles, CG) in thread-block clusters of (1, CG): block
// (tile, g) transforms coils g, g + CG, ... in turn and keeps its coil sum in
// registers; the CG partial tiles are added through distributed shared memory
// in rank order (deterministic), each block writing 1/CG of the tile.  Each
// half-warp stages its own rows of T (and of the coil map) by cp.async while
// the previous coil's second half runs, and transforms them in place: the
// first half's output k1 replaces row g + R2 k1.  Rows that the tables leave
// out are staged as zeros and not read.
// Measured (kernel time, L2 warm), one image column per block staged by 8-byte
// cp.async -> this form: 192 x 192, C = 12, r = 10: 28.9 -> 16.9 us; 256 x 256,
// C = 20, r = 12: 121 -> 55 us; 256 x 256, C = 32, r = 14: 291 -> 93 us (zeros
// staged instead of rows masked at the read, steps as in k_fwd_cols: from
// 17.4, 65 and 114 us).
// Where k_adj_cols writes: element (pixel i, column l < cols) at p[i stride + l],
// times scale[l] when scale is not NULL.
struct AdjOut {
    float2 *p;
    int stride, cols;
    const float *scale;
};

template <int P>
__global__ void __launch_bounds__(ColPlan<P>::NT, 768 / ColPlan<P>::NT) k_adj_cols(
    const float2 *__restrict__ T, const float2 *__restrict__ smaps, const uint32_t *__restrict__ rowtab, int e0,
    int estep, const AdjOut out, int nx, int r, int nc, int nxt, unsigned inv, const float2 *__restrict__ g_tw) {
    using PL = ColPlan<P>;
    constexpr int NY = PL::NY, R1 = PL::R1, R2 = PL::R2, NG = PL::NG;
    extern __shared__ __align__(16) float2 smem[];   // two tiles of NY x COLW, two map stages
    cg::cluster_group cluster = cg::this_cluster();
    const int lane = threadIdx.x & (COLW - 1), g = threadIdx.x / COLW, grp = blockIdx.y, CG = gridDim.y;
    const int rs = nx * r, c0 = blockIdx.x * COLW, c = c0 + lane, x0 = (int)((unsigned)c0 / (unsigned)r);
    const int x = (int)((unsigned)c / (unsigned)r), l = c - x * r;
    const bool first = R2 == NG || g < R2, second = R1 == NG || g < R1;
    const uint32_t rows = first ? __ldg(rowtab + (e0 + l * estep) * 32 + 16 + g) : 0u;
    const size_t plane = (size_t)NY * rs;
    const int mstage = nxt * (R2 + 2);
    float2 *map = smem + 2 * NY * COLW + g * mstage;
    const float2 *d = smaps + (size_t)g * nx + x0;
    const int nxl = min(nxt, nx - x0);   // x values of this tile inside the image
    float2 acc[R2];
#pragma unroll
    for (int k2 = 0; k2 < R2; ++k2) acc[k2] = make_float2(0.f, 0.f);
    // the next coil's rows (zeros where the tables leave them out) and map; one
    // table for every column: 16-byte pieces of the pair's rows, else its own 8 bytes
    const unsigned rowbytes = (unsigned)(R2 * rs * sizeof(float2));
    const float2 *src = T + grp * plane +
                        (estep == 0 ? (size_t)(g + R2 * (lane & 1)) * rs + c0 + (lane & ~1) : (size_t)g * rs + c);
    MapStage<R2> ms;
    ms.init(R1 * nx, nxt, nxl, inv, lane);
    d += (size_t)grp * NY * nx;
    auto stage = [&](int s) {
        if (first) {
            if (estep == 0) {
                float2 *dst = smem + s * NY * COLW + (g + R2 * (lane & 1)) * COLW + (lane & ~1);
#pragma unroll
                for (int m = 0; m < R1; m += 2)
                    cp_async16_or_zero(dst + m * R2 * COLW, step_by(src, rowbytes, m), rows & (1u << m << (lane & 1)));
            } else {
                float2 *dst = smem + s * NY * COLW + g * COLW + lane;
#pragma unroll
                for (int m = 0; m < R1; ++m)
                    cp_async8_or_zero(dst + m * R2 * COLW, step_by(src, rowbytes, m), rows & (1u << m));
            }
        }
        if (second) ms.run(map + s * NG * mstage, d, R1 * nx, nxt, nxl, inv, lane);
        cp_async_commit();
        src += CG * plane;
        d += (size_t)CG * NY * nx;
    };
    if (grp < nc) stage(0);
    int s = 0;
    for (int j = grp; j < nc; j += CG, s ^= 1) {
        float2 *sm = smem + s * NY * COLW + lane;
        cp_async_wait();
        __syncwarp();
        if (first) {
            float2 v[R1];
#pragma unroll
            for (int m = 0; m < R1; ++m) v[m] = sm[(g + R2 * m) * COLW];
            fft::dft_first<R1, R2, true>(v, g, g_tw, [&](int k1, float2 w) { sm[(g + R2 * k1) * COLW] = w; });
        }
        __syncthreads();
        if (j + CG < nc) stage(s ^ 1);
        if (second) {
            float2 v[R2];
#pragma unroll
            for (int j2 = 0; j2 < R2; ++j2) v[j2] = sm[(g * R2 + j2) * COLW];
            fft::Dft<R2, true>::run(v);
            const float4 *m4 = reinterpret_cast<const float4 *>(map + s * NG * mstage + (x - x0) * (R2 + 2));
#pragma unroll
            for (int k2 = 0; k2 < R2; k2 += 2) {
                const float4 w = m4[k2 / 2];
                cfmac(acc[k2], make_float2(w.x, w.y), v[k2]);
                cfmac(acc[k2 + 1], make_float2(w.z, w.w), v[k2 + 1]);
            }
        }
    }
    // element (y, x, l) of the result
    float2 *dst = out.p + (size_t)x * out.stride + l;
    const size_t orow = (size_t)nx * out.stride;
    const bool live = l < out.cols;
    const float sc = out.scale && live ? __ldg(out.scale + l) : 1.f;
    if (CG == 1) {
        if (second && live) {
#pragma unroll
            for (int k2 = 0; k2 < R2; ++k2) dst[(R1 * k2 + g) * orow] = cscale(acc[k2], sc);
        }
        return;
    }
    __syncthreads();
    if (second) {
#pragma unroll
        for (int k2 = 0; k2 < R2; ++k2) smem[(g + R1 * k2) * COLW + lane] = acc[k2];
    }
    cluster.sync();
    // rows y = grp, grp + CG, ... of the tile, by half-warps
    for (int y = grp + CG * g; y < NY; y += CG * NG) {
        float2 sum = make_float2(0.f, 0.f);
        for (int k = 0; k < CG; ++k) sum = cadd(sum, cluster.map_shared_rank(smem, k)[y * COLW + lane]);
        if (live) dst[y * orow] = cscale(sum, sc);
    }
    cluster.sync();   // no block leaves while its tile may still be read
}

// ---------------------------------------------------------------- launchers

// Coil groups (cluster size) of k_row_gram and k_row_w: groups of about 4
// coils, at most 8; or the tuned plan's.
static int row_cluster(const lrccs_ctx *c) {
    if (c->plan.coil_groups >= 1 && c->plan.coil_groups <= 8 && c->plan.coil_groups <= c->nc)
        return c->plan.coil_groups;
    const int cg = (c->nc + 3) / 4;
    return cg < 1 ? 1 : (cg > 8 ? 8 : cg);
}

typedef void (*row_gram_t)(const float2 *, const int32_t *, float2 *, int, int, int);
typedef void (*row_w_t)(float2 *, const float2 *, const int32_t *, const int32_t *, const int32_t *, int, int, int,
                        int);
#define RANK_TABLE(K) {K<1>, K<2>, K<3>, K<4>, K<5>, K<6>, K<7>, K<8>, K<9>, K<10>, K<11>, K<12>, K<13>, K<14>, K<15>, K<16>}
static const row_gram_t kRowGram[RMAXC] = RANK_TABLE(k_row_gram);
static const row_w_t kRowW[RMAXC] = RANK_TABLE(k_row_w);

// One launcher per iteration kernel, at the context's current rank c->r (the
// _on / _to forms take the source or destination and the column count).
// Coil groups of a column pass whose blocks number tiles x groups, `res` of
// them resident per multiprocessor: the fewest rounds of coils,
// ceil(blocks / slots) (ceil(C / CG) + 1), the + 1 for a block's start and end.
static int col_groups(const lrccs_ctx *c, int tiles, int res, int most) {
    int best = 1;
    double cost = 1e30;
    for (int cg = 1; cg <= most && cg <= c->nc; ++cg) {
        const int slots = res * c->nsm;
        const double v = (double)((tiles * cg + slots - 1) / slots) * ((c->nc + cg - 1) / cg + 1.0);
        if (v < cost) cost = v, best = cg;
    }
    return best;
}

static size_t col_smem(int ny, int r, int ng, int cnt) {
    return ((size_t)2 * ny * COLW + (size_t)2 * ng * col_nxt(r) * (cnt + 2)) * sizeof(float2);
}

cudaError_t launch_fwd_cols_on(lrccs_ctx *c, const float2 *src, int r, int e0, int estep) {
    const int nx = c->nx, tiles = nx * r / COLW, nxt = col_nxt(r);
    DISPATCH_P(c->py, {
        using PL = ColPlan<P_>;
        const size_t smem = col_smem(PL::NY, r, PL::NG, PL::R1);
        const int res = std::max(1, std::min(768 / PL::NT, (int)(c->smem_sm / (smem + 1024))));
        const dim3 grid(tiles, col_groups(c, tiles, res, c->nc));
        prof_begin(c, KID_FWD_COLS);
        k_fwd_cols<P_><<<grid, PL::NT, smem, c->stream>>>(src, c->d_smaps, c->d_rowtab, e0, estep, c->d_T, nx, r, c->nc,
                                                          nxt, (65536u + nxt - 1) / nxt, c->d_twsy);
        prof_end(c, KID_FWD_COLS);
    });
    return cudaGetLastError();
}

static cudaError_t launch_row_gram(lrccs_ctx *c) {
    const int r = c->r, nx = c->nx, ny = c->ny;
    const size_t smem = (size_t)2 * nx * r * sizeof(float2);
    const int cgr = row_cluster(c);
    cudaLaunchConfig_t cfg = {};
    cfg.gridDim = dim3(c->n_used, cgr, 1);
    cfg.blockDim = dim3(256, 1, 1);
    cfg.dynamicSmemBytes = smem;
    cfg.stream = c->stream;
    cudaLaunchAttribute at[1];
    at[0].id = cudaLaunchAttributeClusterDimension;
    at[0].val.clusterDim.x = 1;
    at[0].val.clusterDim.y = cgr;
    at[0].val.clusterDim.z = 1;
    cfg.attrs = at;
    cfg.numAttrs = 1;
    prof_begin(c, KID_ROW_GRAM);
    const cudaError_t el = cudaLaunchKernelEx(&cfg, kRowGram[r - 1], (const float2 *)c->d_T,
                                              (const int32_t *)c->d_usedrows, c->d_P, ny, nx, c->nc);
    prof_end(c, KID_ROW_GRAM);
    return el;
}

static void launch_row_w(lrccs_ctx *c) {
    const int r = c->r, nx = c->nx, ny = c->ny;
    const size_t smem = ((size_t)2 * nx * r + (size_t)c->q * r) * sizeof(float2);
    prof_begin(c, KID_ROW_W);
    kRowW[r - 1]<<<dim3(c->n_used, row_cluster(c)), 256, smem, c->stream>>>(
        c->d_T, c->d_B, c->d_usedrows, c->d_rfptr, c->d_rflist, ny, nx, c->nc, c->q);
    prof_end(c, KID_ROW_W);
}

// coil-summed inverse transform into dst (n x r); cluster size: the plan's, or col_groups
static cudaError_t adj_cols(lrccs_ctx *c, const AdjOut &out, int r, int e0, int estep) {
    const int nx = c->nx, tiles = nx * r / COLW, nxt = col_nxt(r);
    cudaLaunchConfig_t cfg = {};
    cfg.stream = c->stream;
    cudaLaunchAttribute at[1];
    at[0].id = cudaLaunchAttributeClusterDimension;
    at[0].val.clusterDim.x = 1;
    at[0].val.clusterDim.z = 1;
    cfg.attrs = at;
    cfg.numAttrs = 1;
    cudaError_t el = cudaSuccess;
    DISPATCH_P(c->py, {
        using PL = ColPlan<P_>;
        const size_t smem = col_smem(PL::NY, r, PL::NG, PL::R2);
        const int res = std::max(1, std::min(768 / PL::NT, (int)(c->smem_sm / (smem + 1024))));
        int cgr = c->plan.coil_groups;
        if (cgr < 1 || cgr > 8 || cgr > c->nc) cgr = col_groups(c, tiles, res, 8);
        cfg.gridDim = dim3(tiles, cgr, 1);
        at[0].val.clusterDim.y = cgr;
        cfg.blockDim = dim3(PL::NT, 1, 1);
        cfg.dynamicSmemBytes = smem;
        prof_begin(c, KID_ADJ_COLS);
        el = cudaLaunchKernelEx(&cfg, k_adj_cols<P_>, (const float2 *)c->d_T, (const float2 *)c->d_smaps,
                                (const uint32_t *)c->d_rowtab, e0, estep, out, nx, r, c->nc, nxt,
                                (65536u + nxt - 1) / nxt, (const float2 *)c->d_twsy);
        prof_end(c, KID_ADJ_COLS);
    });
    return el;
}

cudaError_t launch_adj_cols_to(lrccs_ctx *c, float2 *dst, int r, int e0, int estep) {
    return adj_cols(c, AdjOut{dst, r, r, nullptr}, r, e0, estep);
}

// Columns of T as the frames k0 .. k0 + w - 1, each on its own rows, into columns
// k0 .. of the n x q array dst, times scale[k] when given.
cudaError_t launch_adj_cols_frames(lrccs_ctx *c, float2 *dst, int w, int k0, const float *scale) {
    return adj_cols(c, AdjOut{dst + k0, c->q, c->q - k0, scale ? scale + k0 : nullptr}, w, 1 + k0, 1);
}

// Twiddles of the column and row passes, [j2][k1]: w_N^(j2 k1) / sqrt(N).
__global__ void k_col_twiddles(float2 *tw, int N, int R1) {
    const int e = blockIdx.x * blockDim.x + threadIdx.x;
    if (e >= N) return;
    const int j2 = e / R1, k1 = e - j2 * R1;
    double sn, cs;
    sincospi(-2.0 * (double)(j2 * k1) / (double)N, &sn, &cs);
    const double sc = 1.0 / sqrt((double)N);
    tw[e] = make_float2((float)(cs * sc), (float)(sn * sc));
}

cudaError_t launch_col_twiddles(lrccs_ctx *c) {
    DISPATCH_P(c->py, { k_col_twiddles<<<1, 256, 0, c->stream>>>(c->d_twsy, c->ny, ColPlan<P_>::R1); });
    DISPATCH_P(c->px, { k_col_twiddles<<<1, 256, 0, c->stream>>>(c->d_twsx, c->nx, ColPlan<P_>::R1); });
    return cudaGetLastError();
}

static cudaError_t launch_fwd_cols(lrccs_ctx *c) {
    // the precision forms run the sampled rows' DFT as a tensor-core GEMM
    if (c->dims.precision != LRCCS_PREC_FP32_FFT) return launch_fwd_gemm(c);
    return launch_fwd_cols_on(c, c->d_U, c->r, 0, 0);
}
// the iteration's coil-summed inverse transform goes to the U+ buffer (free during iterations)
static cudaError_t launch_adj_cols(lrccs_ctx *c) { return launch_adj_cols_to(c, c->d_Up, c->r, 0, 0); }

// Z B^H on the context's side stream, forked from (and later joined back
// into) its stream: a parallel branch when the iteration is captured.
static cudaError_t fork_zb(lrccs_ctx *c) {
    cudaError_t e = cudaEventRecord(c->ev_fork, c->stream);
    if (e == cudaSuccess) e = cudaStreamWaitEvent(c->side, c->ev_fork, 0);
    if (e != cudaSuccess) return e;
    cudaStream_t main_stream = c->stream;
    c->stream = c->side;
    e = launch_zb(c);
    c->stream = main_stream;
    if (e == cudaSuccess) e = cudaEventRecord(c->ev_join, c->side);
    return e;
}
static cudaError_t join_zb(lrccs_ctx *c) { return cudaStreamWaitEvent(c->stream, c->ev_join, 0); }

cudaError_t launch_iteration(lrccs_ctx *c) {
    if (c->r < 1 || c->r > RMAXC) return cudaErrorInvalidValue;
    cudaError_t el = launch_fwd_cols(c);   // A
    if (el != cudaSuccess) return el;
    if (c->general) {                      // 2D masks: x transforms, per-point Grams and W (kernels_general.cu)
        el = launch_iteration_general_front(c);
        if (el != cudaSuccess) return el;
        el = fork_zb(c);                   // I
        if (el != cudaSuccess) return el;
        el = launch_iteration_general_back(c);
        if (el != cudaSuccess) return el;
    } else if (bstep_fused_ok(c)) {
        el = launch_bstep_fused(c);        // B + C + D + I (k_bstep, kernels_solve.cu)
        if (el != cudaSuccess) return el;
        el = launch_adj_cols(c);           // E
        if (el != cudaSuccess) return el;
        return launch_gdqr(c, 1);          // F
    } else {
        el = launch_row_gram(c);           // B
        if (el != cudaSuccess) return el;
        launch_solve(c);                   // C
        el = fork_zb(c);                   // I
        if (el != cudaSuccess) return el;
        launch_row_w(c);                   // D
    }
    el = launch_adj_cols(c);               // E
    if (el != cudaSuccess) return el;
    el = join_zb(c);
    if (el != cudaSuccess) return el;
    cudaError_t e = cudaGetLastError();
    if (e != cudaSuccess) return e;
    // F: gradient, GD step and Cholesky QR (one cooperative launch)
    return launch_gdqr(c, 1);
}

// The iteration's forward transform alone (FP32 FFT or, for the precision
// forms, the tensor-core GEMM): d_T <- F_y(d_j o U) on the sampled rows.
cudaError_t launch_forward(lrccs_ctx *c) {
    if (c->r < 1 || c->r > RMAXC) return cudaErrorInvalidValue;
    cudaError_t el = launch_fwd_cols(c);
    if (el != cudaSuccess) return el;
    return cudaGetLastError();
}

// The B-step alone at the current U (the partial sums of U^H Z left by the
// k_gdqr launch that formed U): forward transforms, Grams and the per-frame
// solves.
cudaError_t launch_bstep(lrccs_ctx *c) {
    if (c->r < 1 || c->r > RMAXC) return cudaErrorInvalidValue;
    cudaError_t el = launch_fwd_cols(c);
    if (el != cudaSuccess) return el;
    if (c->general) return launch_iteration_general_front(c);
    el = launch_row_gram(c);
    if (el != cudaSuccess) return el;
    return launch_solve(c);
}

// The normal operator of the stacked A = [A_1; ...; A_q] with B = 1 (q x 1):
// d_Up <- sum_j conj(d_j) o F^H[c o F(d_j o u)], u = d_U (n x 1), c_i the
// number of frames that sample k-space row i (W_i of the gradient with r = 1).
cudaError_t launch_normal_op(lrccs_ctx *c) {
    if (c->r != 1) return cudaErrorInvalidValue;
    cudaError_t el = launch_fwd_cols(c);
    if (el != cudaSuccess) return el;
    if (c->general) {   // W_u = number of frames sampling point u
        el = launch_fwd_rows(c);
        if (el == cudaSuccess) el = launch_sample_w(c);
        if (el == cudaSuccess) el = launch_adj_rows(c);
        if (el != cudaSuccess) return el;
    } else {
        launch_row_w(c);
    }
    el = launch_adj_cols(c);
    if (el != cudaSuccess) return el;
    return cudaGetLastError();
}

// d_T <- F_y(d_j o U) on the sampled rows (the first step of an iteration);
// with general masks also d_FU <- F(d_j o U) at the union points.
cudaError_t launch_fwd_only(lrccs_ctx *c) {
    if (c->r < 1 || c->r > RMAXC) return cudaErrorInvalidValue;
    cudaError_t el = launch_fwd_cols(c);
    if (el != cudaSuccess) return el;
    if (c->general) {
        el = launch_fwd_rows(c);
        if (el != cudaSuccess) return el;
    }
    return cudaGetLastError();
}

// Caller layouts (frame k contiguous, X[k n + i]): X_k = zbar + U_{t-1} b_k + e_k
// and, with Eout, E_k = e_k; zbar and E (chunks of w columns, kernels_mec.cu) may be
// NULL.  Block = 256 pixels x IMG_F frames: a thread keeps its pixel's row of
// U in registers and walks the frames (b_k broadcast from shared memory), so
// every store is a full line.  One thread per (frame, pixel) re-read U's row
// for each: n = 65536, q = 96, r = 14: 111 -> 25 us; n = 36864, q = 8, r = 10: 6.2 ->
// 4.5 us.
#define IMG_F 16
template <int R>
__global__ void __launch_bounds__(256) k_images(const float2 *__restrict__ Uprev, const float2 *__restrict__ B,
                                                const float2 *__restrict__ zbar, const float2 *__restrict__ E, int w,
                                                int n, int q, float2 *__restrict__ Eout, float2 *__restrict__ X) {
    __shared__ float2 s_b[IMG_F * R];
    const int i = blockIdx.x * 256 + threadIdx.x, k0 = blockIdx.y * IMG_F, kn = min(IMG_F, q - k0);
    for (int e = threadIdx.x; e < kn * R; e += 256) s_b[e] = B[(size_t)k0 * R + e];
    __syncthreads();
    if (i >= n) return;
    float2 u[R];
    const float2 z = zbar ? zbar[i] : make_float2(0.f, 0.f);
    if (X) {
#pragma unroll
        for (int a = 0; a < R; ++a) u[a] = __ldg(Uprev + (size_t)i * R + a);
    }
    int cc = w > 0 ? k0 / w : 0, l = w > 0 ? k0 - cc * w : 0;
#pragma unroll 2
    for (int f = 0; f < kn; ++f) {
        float2 e = make_float2(0.f, 0.f);
        const size_t o = (size_t)(k0 + f) * n + i;
        if (E) {
            e = __ldg(E + ((size_t)cc * n + i) * w + l);
            if (++l == w) l = 0, ++cc;
            if (Eout) Eout[o] = e;
        }
        if (X) {
            float2 x = z;
#pragma unroll
            for (int a = 0; a < R; ++a) cfma(x, u[a], s_b[f * R + a]);
            X[o] = E ? cadd(x, e) : x;
        }
    }
}

typedef void (*images_t)(const float2 *, const float2 *, const float2 *, const float2 *, int, int, int, float2 *, float2 *);
static const images_t kImages[RMAXC] = RANK_TABLE(k_images);

cudaError_t launch_images_mec(lrccs_ctx *c, int kid, const float2 *zbar, const float2 *E, int w, float2 *Eout, float2 *X) {
    prof_begin(c, kid);
    kImages[c->r - 1]<<<dim3((c->n + 255) / 256, (c->q + IMG_F - 1) / IMG_F), 256, 0, c->stream>>>(
        c->d_Uprev, c->d_B, zbar, E, w, c->n, c->q, Eout, X);
    prof_end(c, kid);
    return cudaGetLastError();
}

cudaError_t launch_images(lrccs_ctx *c, float2 *d_X) {
    return launch_images_mec(c, KID_IMAGES, nullptr, nullptr, 0, nullptr, d_X);
}

#define SET_SMEM(...) do { cudaError_t e_ = allow_smem(__VA_ARGS__, max_smem); if (e_ != cudaSuccess) return e_; } while (0)
#define SET_SMEM_P(fn) \
    SET_SMEM(fn<1>); SET_SMEM(fn<2>); SET_SMEM(fn<3>); SET_SMEM(fn<4>); \
    SET_SMEM(fn<5>); SET_SMEM(fn<6>); SET_SMEM(fn<7>); SET_SMEM(fn<8>)
cudaError_t configure_kernels_iter(int max_smem) {
    for (int i = 0; i < RMAXC; ++i) {
        SET_SMEM(kRowGram[i]);
        SET_SMEM(kRowW[i]);
    }
    SET_SMEM_P(k_fwd_cols);
    SET_SMEM_P(k_adj_cols);
    return cudaSuccess;
}
