// kernels_init.cu -- spectral initialisation of auto-altGDmin (Alg. 2, init)
// on sm_103a: mask compaction, gamma, Z = [A_k^H y_k], truncated X0, the q x q
// Gram X0^H X0 with a Jacobi eigensolver, and U_0 = X0 V_r Sigma_r^{-1}.
#include <math.h>

#include <algorithm>

#include "common.cuh"
#include "fft.cuh"
#include "internal.h"

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

// ---------------------------------------------------------------- twiddles

__global__ void k_twiddles(float2 *tw, int N) {
    int t = blockIdx.x * blockDim.x + threadIdx.x;
    if (t < N) {
        double s, c;
        sincospi(-2.0 * (double)t / (double)N, &s, &c);  // exp(-2 pi i t / N)
        tw[t] = make_float2((float)c, (float)s);
    }
}

cudaError_t launch_twiddles(float2 *tw, int N, cudaStream_t s) {
    k_twiddles<<<(N + 255) / 256, 256, 0, s>>>(tw, N);
    return cudaGetLastError();
}

// ---------------------------------------------------------------- mask compaction
// Sampling H_k (Sec. II-A) given as a q x n bitmap, any mask: one whose every row
// is fully sampled or empty (1D Cartesian lines) takes the line path, any other the
// general one (meta[MT_GENERAL]).

__global__ void k_rowcount(const uint8_t *__restrict__ mask, int rows, int nx, int32_t *rowcnt) {
    const int w = (blockIdx.x * blockDim.x + threadIdx.x) >> 5;
    const int lane = threadIdx.x & 31;
    if (w >= rows) return;
    const uint8_t *m = mask + (size_t)w * nx;
    int c = 0;
    for (int x = lane; x < nx; x += 32) c += (m[x] != 0);
#pragma unroll
    for (int o = 16; o > 0; o >>= 1) c += __shfl_xor_sync(0xffffffffu, c, o);
    if (lane == 0) rowcnt[w] = c;
}

// Per-frame and per-row structure of the masks from the per-(frame, row)
// sample counts.  Rows of a frame with at least one sample are the frame's
// "frame rows" (its lines, for 1D Cartesian masks): lineptr /
// framerows.  Also the frames' sample counts m_k and offsets fpk (checked
// against the caller's frame_ptr), each (frame, row)'s first sample rowoff, the
// rows sampled by some frame, meta[MT_GENERAL] = 1 when some row is only
// partly sampled (a general 2D mask), and the column passes' row tables
// (kernels_iter.cu): entry 0 the rows some frame samples, entry 1 + k those of
// frame k, then 16 empty entries; [e][g] bit i = row g + R1 i, [e][16 + g] bit i =
// row g + R2 i.
//
// One block of 1024 threads with the counts in shared memory; a warp per frame
// (lanes over the rows, ballot and shuffle prefixes), then a warp per row.
// The chain of dependent global loads bounded the earlier thread-per-frame
// form: 45 us (48 frames of 192 rows) -> 24 us with the column tables, 90 us (96 of
// 256) -> 46 us.
#define ST_NT 1024
LRCCS_DEV int warp_excl_sum(int v, int lane, int &total) {   // exclusive prefix over the warp, and its total
    int x = v;
#pragma unroll
    for (int o = 1; o < 32; o <<= 1) {
        const int t = __shfl_up_sync(0xffffffffu, x, o);
        if (lane >= o) x += t;
    }
    total = __shfl_sync(0xffffffffu, x, 31);
    return x - v;
}
__global__ void __launch_bounds__(ST_NT) k_structure(
    const int32_t *__restrict__ rowcnt, const int64_t *__restrict__ fp_user, int q, int ny, int nx, int R1, int R2,
    int32_t *framerows, int32_t *lineptr, int32_t *rfptr, int32_t *rflist, int32_t *usedrows, int32_t *mks,
    int32_t *fpk, int32_t *rowoff, uint32_t *rowtab, float *xs, int32_t *meta, unsigned int *status, double *scal) {
    extern __shared__ int16_t s_cnt[];   // q x ny (a count is at most nx <= 256)
    __shared__ int s_lines[129], s_fp[129], s_rf[257], s_nu[257];
    __shared__ int s_partial, s_min, s_max, s_total;
    const int tid = threadIdx.x, lane = tid & 31, warp = tid >> 5, nw = ST_NT / 32;
    if (tid == 0) {
        s_partial = 0;
        s_min = 0x7fffffff;
        s_max = 0;
    }
    for (int e = tid; e < q * ny; e += ST_NT) s_cnt[e] = (int16_t)rowcnt[e];
    __syncthreads();
    for (int k = warp; k < q; k += nw) {          // line and sample counts of frame k
        int L = 0, m = 0, part = 0;
        for (int ky = lane; ky < ny; ky += 32) {
            const int c = s_cnt[k * ny + ky];
            L += c > 0;
            m += c;
            part |= (c != 0 && c != nx);
        }
#pragma unroll
        for (int o = 16; o > 0; o >>= 1) {
            L += __shfl_xor_sync(0xffffffffu, L, o);
            m += __shfl_xor_sync(0xffffffffu, m, o);
            part |= __shfl_xor_sync(0xffffffffu, part, o);
        }
        if (lane == 0) {
            s_lines[k] = L;
            s_fp[k] = m;
            mks[k] = m;
            atomicMin(&s_min, m);
            atomicMax(&s_max, m);
            if (part) s_partial = 1;
        }
    }
    for (int ky = warp; ky < ny; ky += nw) {      // frames that sample row ky
        int c = 0;
        for (int k = lane; k < q; k += 32) c += s_cnt[k * ny + ky] > 0;
#pragma unroll
        for (int o = 16; o > 0; o >>= 1) c += __shfl_xor_sync(0xffffffffu, c, o);
        if (lane == 0) s_rf[ky] = c;
    }
    __syncthreads();
    if (warp == 0) {                              // prefixes over the frames (q <= 128)
        int acc = 0, accm = 0;
        for (int k0 = 0; k0 < q; k0 += 32) {
            const int k = k0 + lane;
            int tl, tm;
            const int el = warp_excl_sum(k < q ? s_lines[k] : 0, lane, tl);
            const int em = warp_excl_sum(k < q ? s_fp[k] : 0, lane, tm);
            __syncwarp();
            if (k < q) {
                s_lines[k] = acc + el;
                s_fp[k] = accm + em;
                lineptr[k] = acc + el;
                fpk[k] = accm + em;
                if (fp_user[k] != (int64_t)(accm + em)) atomicOr(status, (unsigned)ST_FRAMEPTR_MISMATCH);
            }
            acc += tl;
            accm += tm;
        }
        if (lane == 0) {
            lineptr[q] = acc;
            fpk[q] = accm;
            s_total = accm;
            meta[MT_NLINES] = acc;
            meta[MT_MMIN] = s_min;
            meta[MT_MMAX] = s_max;
            meta[MT_TOTAL] = accm;
            meta[MT_GENERAL] = s_partial;
            scal[SC_MBAR] = (double)accm / (double)q;
            if (fp_user[q] != (int64_t)accm) atomicOr(status, (unsigned)ST_FRAMEPTR_MISMATCH);
        }
    } else if (warp == 1) {                       // prefixes over the rows
        int acc = 0, nu = 0;
        for (int y0 = 0; y0 < ny; y0 += 32) {
            const int ky = y0 + lane;             // ny is a multiple of 32
            int t, tu;
            const int c = s_rf[ky];
            const int e = warp_excl_sum(c, lane, t), eu = warp_excl_sum(c > 0, lane, tu);
            s_rf[ky] = acc + e;
            s_nu[ky] = c > 0 ? nu + eu : -1;
            rfptr[ky] = acc + e;
            acc += t;
            nu += tu;
        }
        if (lane == 0) {
            rfptr[ny] = acc;
            meta[MT_NUSED] = nu;
        }
    }
    __syncthreads();
    if (tid < q) {                                // X0's column scale 1 / sqrt(m_k mbar)
        const int m = (tid + 1 < q ? s_fp[tid + 1] : s_total) - s_fp[tid];
        xs[tid] = m > 0 ? (float)(1.0 / sqrt((double)m * ((double)s_total / (double)q))) : 0.f;
    }
    for (int k = warp; k < q; k += nw) {          // frame k's rows, in order
        int i = s_lines[k], off = s_fp[k];
        for (int y0 = 0; y0 < ny; y0 += 32) {
            const int ky = y0 + lane, e = k * ny + ky, c = s_cnt[e];
            int tl, tm;
            const int el = warp_excl_sum(c > 0, lane, tl), em = warp_excl_sum(c, lane, tm);
            rowoff[e] = off + em;
            if (c > 0) framerows[i + el] = ky;
            i += tl;
            off += tm;
        }
    }
    for (int ky = warp; ky < ny; ky += nw) {      // the frames of row ky, in order
        int base = s_rf[ky];
        if (lane == 0 && s_nu[ky] >= 0) usedrows[s_nu[ky]] = ky;
        for (int k0 = 0; k0 < q; k0 += 32) {
            const int k = k0 + lane;
            const bool in = k < q && s_cnt[k * ny + ky] > 0;
            const unsigned bal = __ballot_sync(0xffffffffu, in);
            if (in) rflist[base + __popc(bal & ((1u << lane) - 1u))] = k;
            base += __popc(bal);
        }
    }
    for (int e = tid; e < (q + 17) * 32; e += ST_NT) {
        const int en = e >> 5, t = e & 31, g = t & 15, step = t < 16 ? R1 : R2, cnt = t < 16 ? R2 : R1;
        uint32_t bits = 0;
        if (g < step && en <= q)
            for (int i = 0; i < cnt; ++i) {
                const int y = g + step * i;
                const bool used = en == 0 ? s_nu[y] >= 0 : s_cnt[(en - 1) * ny + y] > 0;
                bits |= (uint32_t)used << i;
            }
        rowtab[e] = bits;
    }
}

__global__ void k_fill_idx(const int32_t *__restrict__ framerows, int nx, int32_t *idx) {
    const int g = blockIdx.x;
    const int ky = framerows[g];
    for (int kx = threadIdx.x; kx < nx; kx += blockDim.x) idx[(size_t)g * nx + kx] = ky * nx + kx;
}

cudaError_t launch_compact(lrccs_ctx *c, const uint8_t *d_mask, const int64_t *d_fp_user) {
    const int rows = c->q * c->ny;
    prof_begin(c, KID_ROWCOUNT);
    k_rowcount<<<(rows * 32 + 255) / 256, 256, 0, c->stream>>>(d_mask, rows, c->nx, c->d_rowcnt);
    prof_end(c, KID_ROWCOUNT);
    prof_begin(c, KID_STRUCTURE);
    DISPATCH_P(c->py, {
        using PL = fft::Plan<32 * P_>;
        k_structure<<<1, ST_NT, (size_t)c->q * c->ny * sizeof(int16_t), c->stream>>>(
            c->d_rowcnt, d_fp_user, c->q, c->ny, c->nx, PL::R1, PL::R2, c->d_framerows, c->d_lineptr, c->d_rfptr,
            c->d_rflist, c->d_usedrows, c->d_mks, c->d_fpk, c->d_rowoff, c->d_rowtab, c->d_xs, c->d_meta, c->d_status,
            c->d_scal);
    });
    prof_end(c, KID_STRUCTURE);
    return cudaGetLastError();
}

// Sample indices of masks that are unions of full lines (meta[MT_GENERAL] = 0).
cudaError_t launch_fill_lines(lrccs_ctx *c) {
    prof_begin(c, KID_FILL_IDX);
    k_fill_idx<<<c->n_lines, 128, 0, c->stream>>>(c->d_framerows, c->nx, c->d_idx);
    prof_end(c, KID_FILL_IDX);
    return cudaGetLastError();
}

// ---------------------------------------------------------------- gamma
// gamma = trunc * sum |y|^2 / (number of measured entries)  (Alg. 2, init).
// FP64 adds bound an FP64 sum here (two a cycle per multiprocessor: 50 us for
// 2.7 M entries, 403 us for 34 M), so each thread sums in FP32 without error:
// fsum3 (common.cuh); threads and blocks add in FP64 in a fixed order: 17 us and
// 93 us.

__global__ void __launch_bounds__(256) k_energy(const float2 *__restrict__ y, int64_t count, double trunc, double *part,
                                                unsigned int *counter, double *scal) {
    __shared__ double s_red[8];
    fsum3 s = {0.f, 0.f, 0.f};
    double wide = 0.0;
    const int64_t step = (int64_t)gridDim.x * blockDim.x;
    int64_t i = (int64_t)blockIdx.x * blockDim.x + threadIdx.x;
    for (; i + 3 * step < count; i += 4 * step) {
        float2 v[4];
#pragma unroll
        for (int u = 0; u < 4; ++u) v[u] = __ldg(y + i + u * step);
#pragma unroll
        for (int u = 0; u < 4; ++u) {
            fsum3_mul(s, wide, v[u].x, v[u].x);
            fsum3_mul(s, wide, v[u].y, v[u].y);
        }
    }
    for (; i < count; i += step) {
        const float2 v = __ldg(y + i);
        fsum3_mul(s, wide, v.x, v.x);
        fsum3_mul(s, wide, v.y, v.y);
    }
    const double acc = warp_sum_d(wide + fsum3_total(s));
    if ((threadIdx.x & 31) == 0) s_red[threadIdx.x >> 5] = acc;
    __syncthreads();
    if (threadIdx.x == 0) {
        double b = 0.0;
        for (int w = 0; w < 8; ++w) b += s_red[w];
        part[blockIdx.x] = b;
    }
    if (last_block_arrive(counter) && threadIdx.x < 32) {
        double e = 0.0;
        for (int b = threadIdx.x; b < (int)gridDim.x; b += 32) e += __ldcg(part + b);
        e = warp_sum_d(e);
        if (threadIdx.x == 0) scal[SC_GAMMA] = trunc * e / (double)count;
    }
}

cudaError_t launch_energy(lrccs_ctx *c, const float2 *d_y) {
    const int64_t count = (int64_t)c->nc * c->total;
    const int blocks = 4 * c->nsm < 1024 ? 4 * c->nsm : 1024;   // partials: doubles of d_gpart (at least 1024)
    prof_begin(c, KID_ENERGY);
    k_energy<<<blocks, 256, 0, c->stream>>>(d_y, count, c->prm.trunc_factor, (double *)c->d_gpart,
                                            c->d_counters + CNT_ENERGY, c->d_scal);
    prof_end(c, KID_ENERGY);
    return cudaGetLastError();
}

// ---------------------------------------------------------------- Z and X0
// Z[:, k] = A_k^H y_k and X0[:, k] = A_k^H y_k,tnc / sqrt(m_k mbar) (the plain and
// the truncated data), w frames at a time as the columns of one transform: a
// row pass scatters the frames' samples of k-space row ky and transforms them
// back along x into T[j][ky][x][l] (frame k0 + l), and the iteration's adjoint
// column pass, reading for column l only the rows frame k0 + l samples, does the
// rest and writes column k0 + l of Z or X0.  Any mask takes this path (full
// lines only make the scatter the identity).  Z and X0, kernel time: 16 spokes on
// 256 x 256, q = 64, C = 20: direct sums over each row's samples in one kernel 3.22 ms
// -> 8 chunks of 108 + 89 us; 8 frames of 224 x 224 (Z alone): 0.98 ms -> 26 + 50 us;
// lines of 192 x 192, q = 48, C = 12: 36 + 175 us -> 6 chunks of 15 + 23 us.
//
// Row pass: block (row ky, coil group); only the nf frames of the chunk that
// sample ky take part.  Item (frame c, g): its length-R1 DFT takes kx = g + R2 m
// (lanes along g: contiguous samples), its length-R2 DFT gives x = g + R1 k2
// (lanes along c: neighbouring columns of T).  The exchange tile holds (k1, c,
// j2) at k1 S + c (R2 + 1) + j2, S = nf modulo 16, free of bank conflicts on both
// sides; samples are staged in place one coil step ahead, as in the general
// row passes.
struct InitArgs {
    const float2 *y;
    const int32_t *usedrows, *rfptr, *rflist, *rowoff, *fpk, *mks;
    const uint8_t *mask;       // q x n bitmap (general masks), or NULL: full lines
    const double *scal;
    const float2 *tw;          // [j2][k1] twiddles with the scale 1 / sqrt(nx)
    int ny, nc, w, k0;
};

template <int P>
struct RowPlanI {
    static constexpr int NX = 32 * P, R1 = fft::Plan<NX>::R1, R2 = fft::Plan<NX>::R2, NG = R1 > R2 ? R1 : R2;
    static __host__ __device__ int coils(int nf, int nc) {   // coils at a time: a block of 256 threads
        const int cb = 256 / (NG * nf);
        return cb < 1 ? 1 : (cb < nc ? cb : nc);
    }
    static __host__ __device__ int stride(int nf) { return nf * (R2 + 1) + (16 - nf * R2 % 16) % 16; }
};

template <int P, bool TRUNC>
__global__ void __launch_bounds__(256, 3) k_init_rows(float2 *__restrict__ T, const InitArgs a) {
    using PL = RowPlanI<P>;
    constexpr int NX = PL::NX, R1 = PL::R1, R2 = PL::R2, NG = PL::NG;
    extern __shared__ __align__(16) float2 smem[];
    __shared__ int16_t s_pos[16 * NX];   // general masks: sample index of kx in the frame's row, or -1
    __shared__ int s_fr[16], s_nf;
    __shared__ int64_t s_base[16];       // first sample of (frame, row) for coil 0
    __shared__ int s_m[16];
    const int ky = a.usedrows[blockIdx.x], lane = threadIdx.x & 31, warp = threadIdx.x >> 5;
    if (warp == 0) {
        int nf = 0;
        for (int f0 = a.rfptr[ky]; f0 < a.rfptr[ky + 1]; f0 += 32) {
            const int f = f0 + lane, k = f < a.rfptr[ky + 1] ? a.rflist[f] : -1;
            const bool in = k >= a.k0 && k < a.k0 + a.w;
            const unsigned bal = __ballot_sync(0xffffffffu, in);
            if (in) {
                const int c = nf + __popc(bal & ((1u << lane) - 1u)), f0k = a.fpk[k];
                s_fr[c] = k;
                s_m[c] = a.mks[k];
                s_base[c] = (int64_t)a.nc * f0k + (a.rowoff[k * a.ny + ky] - f0k);
            }
            nf += __popc(bal);
        }
        if (lane == 0) s_nf = nf;
    }
    __syncthreads();
    const int nf = s_nf;
    if (nf == 0) return;   // the same for every thread of the block
    if (a.mask) {
        for (int c = warp; c < nf; c += 8) {
            const uint8_t *m = a.mask + ((size_t)s_fr[c] * a.ny + ky) * NX;
            int pos = 0;
            for (int x0 = 0; x0 < NX; x0 += 32) {
                const bool in = m[x0 + lane] != 0;
                const unsigned bal = __ballot_sync(0xffffffffu, in);
                s_pos[c * NX + x0 + lane] = (int16_t)(in ? pos + __popc(bal & ((1u << lane) - 1u)) : -1);
                pos += __popc(bal);
            }
        }
        __syncthreads();
    }
    const int CB = PL::coils(nf, a.nc), IT = NG * nf, S = PL::stride(nf), tile = R1 * S;
    const int slot = threadIdx.x / IT, i = threadIdx.x - slot * IT;
    const int c1 = i / NG, g1 = i - c1 * NG, g2 = i / nf, c2 = i - g2 * nf;
    const bool first = slot < CB && g1 < R2, second = slot < CB && g2 < R1;
    const int step = gridDim.y * CB;
    float2 *mine = smem + slot * tile;
    uint32_t bits = 0;
    if (first) {
        bits = (1u << R1) - 1u;
        if (a.mask) {
            bits = 0;
            for (int m = 0; m < R1; ++m) bits |= (uint32_t)(s_pos[c1 * NX + g1 + R2 * m] >= 0) << m;
        }
    }
    auto stage = [&](int j, int s) {
        if (bits != 0 && j < a.nc) {
            float2 *dst = mine + s * CB * tile + c1 * (R2 + 1) + g1;
            const float2 *src = a.y + s_base[c1] + (int64_t)j * s_m[c1];
#pragma unroll
            for (int m = 0; m < R1; ++m)
                if (bits >> m & 1) cp_async8(dst + m * S, src + (a.mask ? (int)s_pos[c1 * NX + g1 + R2 * m] : g1 + R2 * m));
        }
        cp_async_commit();
    };
    stage(blockIdx.y * CB + slot, 0);
    const double gam = TRUNC ? a.scal[SC_GAMMA] : 0.0;
    const float glo = (float)(gam * (1.0 - 1e-5)), ghi = (float)(gam * (1.0 + 1e-5));
    int s = 0;
    for (int b = blockIdx.y * CB; b < a.nc; b += step, s ^= 1) {
        const int j = b + slot;
        float2 *ex = mine + s * CB * tile;
        cp_async_wait();
        if (first && j < a.nc) {
            float2 v[R1], *e = ex + c1 * (R2 + 1) + g1;
#pragma unroll
            for (int m = 0; m < R1; ++m) {
                v[m] = (bits >> m & 1) ? e[m * S] : make_float2(0.f, 0.f);
                if (TRUNC && trunc_drop(v[m], gam, glo, ghi)) v[m] = make_float2(0.f, 0.f);
            }
            fft::dft_first<R1, R2, true>(v, g1, a.tw, [&](int k1, float2 w) { e[k1 * S] = w; });
        }
        __syncthreads();
        if (b + step < a.nc) stage(j + step, s ^ 1);
        if (second && j < a.nc) {
            float2 v[R2];
            const float2 *e = ex + g2 * S + c2 * (R2 + 1);
#pragma unroll
            for (int j2 = 0; j2 < R2; ++j2) v[j2] = e[j2];
            fft::Dft<R2, true>::run(v);
            float2 *dst = T + (((size_t)j * a.ny + ky) * NX + g2) * a.w + (s_fr[c2] - a.k0);
#pragma unroll
            for (int k2 = 0; k2 < R2; ++k2) dst[(size_t)(R1 * k2) * a.w] = v[k2];
        }
    }
}

template <int P>
static cudaError_t launch_init_rows(lrccs_ctx *c, const float2 *d_y, int w, int k0, bool trunc) {
    using PL = RowPlanI<P>;
    InitArgs a;
    a.y = d_y;
    a.usedrows = c->d_usedrows;
    a.rfptr = c->d_rfptr;
    a.rflist = c->d_rflist;
    a.rowoff = c->d_rowoff;
    a.fpk = c->d_fpk;
    a.mks = c->d_mks;
    a.mask = c->general ? c->d_maskc : nullptr;
    a.scal = c->d_scal;
    a.tw = c->d_twsx;
    a.ny = c->ny;
    a.nc = c->nc;
    a.w = w;
    a.k0 = k0;
    size_t tile = 0;   // two tiles of the widest row the chunk can hold
    for (int nf = 1; nf <= w; ++nf) tile = std::max(tile, (size_t)PL::coils(nf, c->nc) * PL::R1 * PL::stride(nf));
    const dim3 grid(c->n_used, std::max(1, std::min(c->nc, (4 * c->nsm + c->n_used - 1) / c->n_used)));
    prof_begin(c, KID_INIT_ROWS);
    if (trunc) k_init_rows<P, true><<<grid, 256, 2 * tile * sizeof(float2), c->stream>>>(c->d_T, a);
    else k_init_rows<P, false><<<grid, 256, 2 * tile * sizeof(float2), c->stream>>>(c->d_T, a);
    prof_end(c, KID_INIT_ROWS);
    return cudaGetLastError();
}

// Z, and with trunc also X0.
cudaError_t launch_init_adjoint(lrccs_ctx *c, const float2 *d_y, bool trunc) {
    const int wmax = (int)std::min<size_t>(16, c->T_cap / ((size_t)c->nc * c->n));
    const int nch = (c->q + wmax - 1) / wmax, w = (c->q + nch - 1) / nch;
    for (int ch = 0; ch < (trunc ? 2 : 1); ++ch)
        for (int k0 = 0; k0 < c->q; k0 += w) {
            DISPATCH_P(c->px, {
                cudaError_t e = launch_init_rows<P_>(c, d_y, w, k0, ch == 1);
                if (e != cudaSuccess) return e;
            });
            // X0's columns are scaled by 1 / sqrt(m_k mbar)
            cudaError_t e = launch_adj_cols_frames(c, ch ? c->d_X0 : c->d_Z, w, k0, ch ? c->d_xs : nullptr);
            if (e != cudaSuccess) return e;
        }
    return cudaSuccess;
}

// ---------------------------------------------------------------- Gram of X0 and its eigensolver

// X0^H X0: thread (4 x 4 tile of frame pairs on or above the diagonal, pixel
// slice) adds its 16 products per pixel from four 16-byte reads; the slices of a
// tile add in order at the end.  Two 8-byte reads per product bounded one pair
// per item: 36864 x 48: 60 -> 25 us, 65536 x 64: 152 -> 63 us.
#define GRAM_CHUNK 32
#define GRAM_THREADS 512

__host__ __device__ inline int gram_tiles(int q) { const int t = (q + 3) / 4; return t * (t + 1) / 2; }
__host__ __device__ inline int gram_slices(int q) {   // pixel slices per tile
    const int t = gram_tiles(q), s = GRAM_THREADS / t;
    return t >= GRAM_THREADS ? 1 : (s < GRAM_CHUNK ? s : GRAM_CHUNK);
}

template <int NS>   // tiles per thread: gram_tiles(q) <= GRAM_THREADS NS
__global__ void __launch_bounds__(GRAM_THREADS) k_gram_x0(const float2 *__restrict__ X0, int n, int q, float2 *part) {
    extern __shared__ __align__(16) float2 s_x[];   // GRAM_CHUNK x qp (columns past q zero), then the slices' sums
    const int nt = (q + 3) / 4, qp = 4 * nt + 2, T = gram_tiles(q), S = gram_slices(q);
    const int per = (n + gridDim.x - 1) / gridDim.x;
    const int i0 = blockIdx.x * per, i1 = min(n, i0 + per);
    const int sl = threadIdx.x / T;
    float2 acc[NS][16];
    int ta[NS], tb[NS];
#pragma unroll
    for (int u = 0; u < NS; ++u) {
        const int w = NS == 1 ? threadIdx.x - sl * T : threadIdx.x + u * GRAM_THREADS;
        int A = 0, B = 0;
        const bool live = NS == 1 ? sl < S : w < T;
        if (live) pair_of(w, nt, A, B);
        ta[u] = live ? 4 * A : -1;
        tb[u] = 4 * B;
#pragma unroll
        for (int m = 0; m < 16; ++m) acc[u][m] = make_float2(0.f, 0.f);
    }
    const int s0 = NS == 1 ? sl : 0, step = NS == 1 ? S : 1;
    for (int c0 = i0; c0 < i1; c0 += GRAM_CHUNK) {
        const int cn = min(GRAM_CHUNK, i1 - c0);
        __syncthreads();
        for (int e = threadIdx.x; e < cn * qp; e += GRAM_THREADS) {
            const int ii = e / qp, k = e - ii * qp;
            s_x[e] = k < q ? __ldg(X0 + (size_t)(c0 + ii) * q + k) : make_float2(0.f, 0.f);
        }
        __syncthreads();
#pragma unroll
        for (int u = 0; u < NS; ++u) {
            if (ta[u] < 0) continue;
            for (int ii = s0; ii < cn; ii += step) {
                const float4 *x4 = reinterpret_cast<const float4 *>(s_x + ii * qp + ta[u]);
                const float4 *y4 = reinterpret_cast<const float4 *>(s_x + ii * qp + tb[u]);
                const float4 xa = x4[0], xb = x4[1], ya = y4[0], yb = y4[1];
                const float2 x[4] = {make_float2(xa.x, xa.y), make_float2(xa.z, xa.w), make_float2(xb.x, xb.y),
                                     make_float2(xb.z, xb.w)};
                const float2 y[4] = {make_float2(ya.x, ya.y), make_float2(ya.z, ya.w), make_float2(yb.x, yb.y),
                                     make_float2(yb.z, yb.w)};
#pragma unroll
                for (int m = 0; m < 16; ++m) cfmac(acc[u][m], x[m >> 2], y[m & 3]);
            }
        }
    }
    // the slices' sums, a row of the tiles at a time, then pair (a, b), a <= b, to part
    float2 *out = part + (size_t)blockIdx.x * (q * (q + 1) / 2);
#pragma unroll
    for (int h = 0; h < 4; ++h) {
        __syncthreads();
#pragma unroll
        for (int u = 0; u < NS; ++u)
#pragma unroll
            for (int x = 0; x < 4; ++x)
                if (ta[u] >= 0) s_x[x * NS * GRAM_THREADS + u * GRAM_THREADS + threadIdx.x] = acc[u][4 * h + x];
        __syncthreads();
        for (int e = threadIdx.x; e < 4 * T; e += GRAM_THREADS) {
            const int x = e / T, w = e - x * T;
            int A, B;
            pair_of(w, nt, A, B);
            const int a = 4 * A + h, b = 4 * B + x;
            if (a > b || b >= q) continue;
            float2 sum = make_float2(0.f, 0.f);
            for (int ss = 0; ss < S; ++ss) sum = cadd(sum, s_x[x * NS * GRAM_THREADS + ss * T + w]);
            out[pair_index(a, b, q)] = sum;
        }
    }
}

// Sum the nblk partial rows of k_gram_x0 into the FP64 Hermitian Gram: thread
// (pair p, slice s of 4) adds blocks s, s + 4, ... in compensated FP32 with 8
// loads in flight; the 4 slices are then added in order.
__global__ void __launch_bounds__(256) k_gram_sum(const float2 *__restrict__ part, int nblk, int q,
                                                  double *__restrict__ gram) {
    __shared__ float4 s_acc[256];
    const int np = q * (q + 1) / 2;
    const int pl = threadIdx.x & 63, sl = threadIdx.x >> 6;
    const int p = blockIdx.x * 64 + pl;
    fsum2 re = {0.f, 0.f}, im = {0.f, 0.f};
    if (p < np) {
        int b = sl;
        for (; b + 28 < nblk; b += 32) {
            float2 v[8];
#pragma unroll
            for (int u = 0; u < 8; ++u) v[u] = __ldcg(part + (size_t)(b + 4 * u) * np + p);
#pragma unroll
            for (int u = 0; u < 8; ++u) {
                fsum_add(re, v[u].x);
                fsum_add(im, v[u].y);
            }
        }
        for (; b < nblk; b += 4) {
            const float2 v = __ldcg(part + (size_t)b * np + p);
            fsum_add(re, v.x);
            fsum_add(im, v.y);
        }
    }
    s_acc[threadIdx.x] = make_float4(re.hi, re.lo, im.hi, im.lo);
    __syncthreads();
    if (sl == 0 && p < np) {
        fsum2 R = {s_acc[pl].x, s_acc[pl].y}, I = {s_acc[pl].z, s_acc[pl].w};
        for (int k = 1; k < 4; ++k) {
            const float4 w = s_acc[k * 64 + pl];
            R = fsum_pair(R, fsum2{w.x, w.y});
            I = fsum_pair(I, fsum2{w.z, w.w});
        }
        int a, bb;
        pair_of(p, q, a, bb);
        const double sr = (double)R.hi + (double)R.lo, si = (double)I.hi + (double)I.lo;
        gram[2 * (a * q + bb)] = sr;
        gram[2 * (a * q + bb) + 1] = si;
        gram[2 * (bb * q + a)] = sr;
        gram[2 * (bb * q + a) + 1] = -si;
    }
}

// Eigendecomposition of the q x q Gram A = X0^H X0 (Alg. 2: sigma_j^2 and the
// right singular vectors of X0) in two passes, each a parallel cyclic Jacobi
// in FP32 in one block:
//   pass 0 : Jacobi on A (rounded to FP32) -> V0.  Its rotations leave errors
//            of about eps ||A|| in every entry, so the eigenvectors of small
//            eigenvalues are off by about eps lambda_1 / gap;
//   refine : B = V0^H A V0 formed in FP64 (k_refine_av, k_refine_vhb), whose
//            off-diagonal entries are those small errors, held in FP32 with
//            full relative precision; a second Jacobi (relative threshold
//            only) on B -> Q, and V = V0 Q.  The second pass's rounding is
//            relative to the entries it rotates, so every eigenpair comes out
//            accurate relative to its own eigenvalue and gap (mixed-precision
//            Jacobi refinement).
// The refine pass also sorts: sigma_j = sqrt(lambda_j) descending, and the
// rank rule of Alg. 2 when rank_in == 0: the smallest r whose leading sigma^2
// reach b% of the energy of the first floor(min(n, q, C min m_k)/10) (at least 1).
__global__ void __launch_bounds__(1024) k_eig(const double *__restrict__ gram, int q, int n, int nc, int rank_in, int rmax,
                      double energy_pct, float2 *V, float2 *Q, int32_t *order, double *sigma, int32_t *meta,
                      unsigned int *status, int v_in_smem, int refine) {
    // A (and the rotation matrix when it fits) in shared memory with an odd row
    // pitch, so that the column updates of the rotations hit distinct banks
    extern __shared__ float2 sA[];
    __shared__ JacobiWork s_jac;
    __shared__ double s_fro[32];
    __shared__ double s_scale;
    __shared__ float s_lam[128];
    const int n2 = jacobi_rows(q), ld = n2 | 1;
    float2 *Vw = v_in_smem ? sA + n2 * ld : (refine ? Q : V);
    const int ldv = v_in_smem ? ld : q;
    if (threadIdx.x < 32) {   // the refine pass works on B / max diag(B)
        double mx = 0.0;
        if (refine)
            for (int i = threadIdx.x; i < q; i += 32) mx = fmax(mx, gram[2 * (i * q + i)]);
        for (int o = 16; o; o >>= 1) mx = fmax(mx, __shfl_xor_sync(0xffffffffu, mx, o));
        if (threadIdx.x == 0) s_scale = mx > 0.0 ? mx : 1.0;
    }
    __syncthreads();
    const double isc = refine ? 1.0 / s_scale : 1.0;
    double fro = 0.0;
    for (int e = threadIdx.x; e < n2 * ld; e += blockDim.x) sA[e] = make_float2(0.f, 0.f);
    __syncthreads();
    for (int e = threadIdx.x; e < q * q; e += blockDim.x) {
        const int a = e / q, b = e - a * q;
        sA[a * ld + b] = make_float2((float)(gram[2 * e] * isc), (float)(gram[2 * e + 1] * isc));
        Vw[a * ldv + b] = make_float2(a == b ? 1.f : 0.f, 0.f);
        fro += gram[2 * e] * gram[2 * e] + gram[2 * e + 1] * gram[2 * e + 1];
    }
    fro = warp_sum_d(fro);
    if ((threadIdx.x & 31) == 0) s_fro[threadIdx.x >> 5] = fro;
    __syncthreads();
    fro = 0.0;
    for (int w = 0; w < (int)(blockDim.x >> 5); ++w) fro += s_fro[w];
    if (!refine) {
        // a rotation is skipped once |a_pq| <= 1e-5 sqrt(a_pp a_qq) or <= 1e-6
        // ||A||_F, at most 5 sweeps: this pass only has to leave B = V0^H A V0
        // diagonally dominant; the refine pass converges quadratically from there
        block_jacobi<true>(sA, q, ld, Vw, ldv, s_jac, 5, (float)(1e-6 * sqrt(fro)), 1e-5f);
        if (v_in_smem)
            for (int e = threadIdx.x; e < q * q; e += blockDim.x) V[e] = Vw[(e / q) * ldv + e % q];
        return;
    }
    // the wanted eigenpairs: the top rank_in (fixed rank) or the rank rule's
    // cap; rotations between two indices whose diagonal entries are both
    // below a quarter of the r_w-th largest entry cannot change them
    __shared__ float s_tail;
    {
        int capn = min(n, q);
        const long long cm = (long long)nc * meta[MT_MMIN];
        if (cm < capn) capn = (int)cm;
        const int cap = max(1, capn / 10);
        const int rw = min(q, max(rank_in, cap));
        for (int i = threadIdx.x; i < q; i += blockDim.x) {
            const float di = sA[i * ld + i].x;
            int above = 0;
            for (int j = 0; j < q; ++j) {
                const float dj = sA[j * ld + j].x;
                above += (dj > di || (dj == di && j < i)) ? 1 : 0;
            }
            if (above == rw - 1) s_tail = 0.25f * di;
        }
        __syncthreads();
    }
    block_jacobi<true>(sA, q, ld, Vw, ldv, s_jac, 6, 0.f, 1e-6f, s_tail);
    // eigenvalues (diagonal of the rotated B, scaled back), then V <- V0 Q,
    // formed in the shared A region (A is no longer needed)
    for (int i = threadIdx.x; i < q; i += blockDim.x) s_lam[i] = sA[i * ld + i].x;
    __syncthreads();
    for (int e = threadIdx.x; e < q * q; e += blockDim.x) {
        const int a = e / q, b = e - a * q;
        float2 acc = make_float2(0.f, 0.f);
        for (int m = 0; m < q; ++m) cfma(acc, V[a * q + m], Vw[m * ldv + b]);
        sA[a * ld + b] = acc;
    }
    __syncthreads();
    for (int e = threadIdx.x; e < q * q; e += blockDim.x) V[e] = sA[(e / q) * ld + e % q];
    // eigenvalue order, descending (ties by index): thread i finds its rank
    for (int i = threadIdx.x; i < q; i += blockDim.x) {
        const float li = s_lam[i];
        int rank = 0;
        for (int j = 0; j < q; ++j) {
            const float lj = s_lam[j];
            rank += (lj > li || (lj == li && j < i)) ? 1 : 0;
        }
        order[rank] = i;
        sigma[rank] = sqrt(li > 0.f ? (double)li * s_scale : 0.0);
    }
    __syncthreads();
    if (threadIdx.x == 0) {
        int r = rank_in;
        if (r <= 0) {
            long long capn = min(n, q);
            long long cm = (long long)nc * meta[MT_MMIN];
            if (cm < capn) capn = cm;
            int cap = (int)(capn / 10);
            if (cap < 1) cap = 1;
            double tot = 0.0, acc = 0.0;
            for (int j = 0; j < cap; ++j) tot += sigma[j] * sigma[j];
            r = cap;
            for (int j = 0; j < cap; ++j) {
                acc += sigma[j] * sigma[j];
                if (acc >= energy_pct / 100.0 * tot) { r = j + 1; break; }
            }
        }
        meta[MT_RANK] = r;
        if (r > rmax || r > q) atomicOr(status, (unsigned)ST_ZERO_SIGMA);
        else if (!(sigma[r - 1] > 0.0)) atomicOr(status, (unsigned)ST_ZERO_SIGMA);
    }
}

// T = A V0 in FP64 (A: the FP64 Gram, (re, im) pairs; V0: FP32 eigenvectors
// of pass 0): block a forms row a of T.
__global__ void k_refine_av(const double *__restrict__ gram, const float2 *__restrict__ V, int q, double *T) {
    const int a = blockIdx.x;
    for (int b = threadIdx.x; b < q; b += blockDim.x) {
        double re = 0.0, im = 0.0;
        for (int j = 0; j < q; ++j) {
            const double ar = gram[2 * (a * q + j)], ai = gram[2 * (a * q + j) + 1];
            const float2 v = V[j * q + b];
            re += ar * v.x - ai * v.y;
            im += ar * v.y + ai * v.x;
        }
        T[2 * (a * q + b)] = re;
        T[2 * (a * q + b) + 1] = im;
    }
}

// B = V0^H T in FP64, made exactly Hermitian (the mean of B and B^H): block a
// forms row a; entries (a, b) and (b, a) are summed in the same order.
__global__ void k_refine_vhb(const float2 *__restrict__ V, const double *__restrict__ T, int q, double *Bm) {
    const int a = blockIdx.x;
    for (int b = threadIdx.x; b < q; b += blockDim.x) {
        double re = 0.0, im = 0.0, re2 = 0.0, im2 = 0.0;
        for (int i = 0; i < q; ++i) {
            const float2 va = V[i * q + a], vb = V[i * q + b];
            const double tr = T[2 * (i * q + b)], ti = T[2 * (i * q + b) + 1];   // T[i][b]
            const double ur = T[2 * (i * q + a)], ui = T[2 * (i * q + a) + 1];   // T[i][a]
            re += va.x * tr + va.y * ti;    // conj(V[i][a]) T[i][b] = B[a][b]
            im += va.x * ti - va.y * tr;
            re2 += vb.x * ur + vb.y * ui;   // conj(V[i][b]) T[i][a] = B[b][a]
            im2 += vb.x * ui - vb.y * ur;
        }
        Bm[2 * (a * q + b)] = 0.5 * (re + re2);
        Bm[2 * (a * q + b) + 1] = 0.5 * (im - im2);
    }
}

cudaError_t launch_gram_x0(lrccs_ctx *c) {
    const int q = c->q;
    const int np = q * (q + 1) / 2;
    int blocks = (c->n + 127) / 128;
    if (blocks > 152) blocks = 152;
    if ((size_t)blocks * np > c->gpart_cap) blocks = (int)(c->gpart_cap / np);
    const int ns = gram_tiles(q) <= GRAM_THREADS ? 1 : 2;
    const size_t smem = std::max(GRAM_CHUNK * (4 * ((q + 3) / 4) + 2), 4 * ns * GRAM_THREADS) * sizeof(float2);
    double *gram = c->d_gram;
    prof_begin(c, KID_GRAM_X0);
    if (ns == 1) k_gram_x0<1><<<blocks, GRAM_THREADS, smem, c->stream>>>(c->d_X0, c->n, q, c->d_gpart);
    else k_gram_x0<2><<<blocks, GRAM_THREADS, smem, c->stream>>>(c->d_X0, c->n, q, c->d_gpart);
    k_gram_sum<<<(np + 63) / 64, 256, 0, c->stream>>>(c->d_gpart, blocks, q, gram);
    prof_end(c, KID_GRAM_X0);
    cudaError_t e = cudaGetLastError();
    if (e != cudaSuccess) return e;
    const int n2 = jacobi_rows(q), ld = n2 | 1;
    const int v_in_smem = (size_t)2 * n2 * ld * sizeof(float2) + sizeof(JacobiWork) + 2048 <= (size_t)c->dev_smem_optin;
    const size_t smem2 = (size_t)(v_in_smem ? 2 : 1) * n2 * ld * sizeof(float2);
    double *T = c->d_gram + 2 * (size_t)q * q, *Bm = T + 2 * (size_t)q * q;
    // one warp a pair for V, as far as 1024 threads go
    const int nthr = std::min(1024, jacobi_block_threads(q) + 32 * std::max(3, (q + 1) / 2));
    prof_begin(c, KID_EIG);
    k_eig<<<1, nthr, smem2, c->stream>>>(gram, q, c->n, c->nc, c->dims.rank, c->rmax, c->prm.energy_pct, c->d_V,
                                        c->d_Q, c->d_meta + MT_COUNT, c->d_sigma, c->d_meta, c->d_status, v_in_smem,
                                        0);
    prof_end(c, KID_EIG);
    prof_begin(c, KID_EIG);
    k_refine_av<<<q, 128, 0, c->stream>>>(gram, c->d_V, q, T);
    prof_end(c, KID_EIG);
    prof_begin(c, KID_EIG);
    k_refine_vhb<<<q, 128, 0, c->stream>>>(c->d_V, T, q, Bm);
    prof_end(c, KID_EIG);
    prof_begin(c, KID_EIG);
    k_eig<<<1, nthr, smem2, c->stream>>>(Bm, q, c->n, c->nc, c->dims.rank, c->rmax, c->prm.energy_pct, c->d_V,
                                        c->d_Q, c->d_meta + MT_COUNT, c->d_sigma, c->d_meta, c->d_status, v_in_smem,
                                        1);
    prof_end(c, KID_EIG);
    return cudaGetLastError();
}

// ---------------------------------------------------------------- U_0
// U_0 = X0 V_r Sigma_r^{-1}: the top-r left singular vectors of X0 (Alg. 2),
// written to the U+ buffer and then orthonormalised by Cholesky QR.  The
// product is k_zb's X0 conj(Q) with Q = conj(V_r Sigma_r^{-1}) (q x r), formed
// here; a thread per entry with both factors re-read took 21 us (36864 x 48, r = 10)
// and 49 us (65536 x 64, r = 12), k_zb 13 and 26 us, both launches.
__global__ void k_u0(const float2 *__restrict__ V, const int32_t *__restrict__ order, const double *__restrict__ sigma,
                     int q, int r, float2 *__restrict__ Q) {
    for (int e = threadIdx.x; e < q * r; e += blockDim.x) {
        const int k = e / r, l = e - k * r;
        Q[e] = cconj(cscale(V[k * q + order[l]], (float)(1.0 / sigma[l])));
    }
}

cudaError_t launch_u0(lrccs_ctx *c) {
    prof_begin(c, KID_U0);
    k_u0<<<1, 256, 0, c->stream>>>(c->d_V, c->d_meta + MT_COUNT, c->d_sigma, c->q, c->r, c->d_B);
    launch_zb_of(c, c->d_X0, c->d_B, c->d_Up);
    prof_end(c, KID_U0);
    return cudaGetLastError();
}

// Allow every kernel of this file the device's opt-in shared memory per block
// (the launch still requests only what it needs).
#define SET_SMEM(...) do { cudaError_t e_ = allow_smem(__VA_ARGS__, max_smem); if (e_ != cudaSuccess) return e_; } while (0)
#define SET_SMEM_B(fn, P) SET_SMEM(fn<P, false>); SET_SMEM(fn<P, true>)
cudaError_t configure_kernels_init(int max_smem) {
    SET_SMEM_B(k_init_rows, 1); SET_SMEM_B(k_init_rows, 2); SET_SMEM_B(k_init_rows, 3); SET_SMEM_B(k_init_rows, 4);
    SET_SMEM_B(k_init_rows, 5); SET_SMEM_B(k_init_rows, 6); SET_SMEM_B(k_init_rows, 7); SET_SMEM_B(k_init_rows, 8);
    SET_SMEM(k_gram_x0<1>); SET_SMEM(k_gram_x0<2>);
    SET_SMEM(k_eig);
    SET_SMEM(k_structure);
    return cudaGetLastError();
}
