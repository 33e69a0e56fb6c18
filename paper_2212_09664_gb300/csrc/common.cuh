// common.cuh -- complex helpers, the warp-level FFT engine and block reductions
// shared by the liblrccs kernels (sm_103a).
#pragma once

#include <cuda_runtime.h>
#include <stdint.h>

#define LRCCS_DEV __device__ __forceinline__

// ---------------------------------------------------------------- complex64

LRCCS_DEV float2 cmul(float2 a, float2 b) { return make_float2(a.x * b.x - a.y * b.y, a.x * b.y + a.y * b.x); }
// conj(a) * b
LRCCS_DEV float2 cmulc(float2 a, float2 b) { return make_float2(a.x * b.x + a.y * b.y, a.x * b.y - a.y * b.x); }
// one packed instruction for both parts (the same two roundings): the transform
// kernels issue an instruction in up to half of their cycles
LRCCS_DEV float2 cadd(float2 a, float2 b) {
    float2 d;
    asm("{\n.reg .b64 a, b, d;\nmov.b64 a, {%2, %3};\nmov.b64 b, {%4, %5};\nadd.rn.f32x2 d, a, b;\n"
        "mov.b64 {%0, %1}, d;\n}\n"
        : "=f"(d.x), "=f"(d.y)
        : "f"(a.x), "f"(a.y), "f"(b.x), "f"(b.y));
    return d;
}
LRCCS_DEV float2 csub(float2 a, float2 b) {
    float2 d;
    asm("{\n.reg .b64 a, b, d;\nmov.b64 a, {%2, %3};\nmov.b64 b, {%4, %5};\nsub.rn.f32x2 d, a, b;\n"
        "mov.b64 {%0, %1}, d;\n}\n"
        : "=f"(d.x), "=f"(d.y)
        : "f"(a.x), "f"(a.y), "f"(b.x), "f"(b.y));
    return d;
}
LRCCS_DEV float2 cconj(float2 a) { return make_float2(a.x, -a.y); }
LRCCS_DEV float2 cscale(float2 a, float s) { return make_float2(a.x * s, a.y * s); }
// acc += a * b
LRCCS_DEV void cfma(float2 &acc, float2 a, float2 b) {
    acc.x = fmaf(a.x, b.x, fmaf(-a.y, b.y, acc.x));
    acc.y = fmaf(a.x, b.y, fmaf(a.y, b.x, acc.y));
}
// acc += conj(a) * b
LRCCS_DEV void cfmac(float2 &acc, float2 a, float2 b) {
    acc.x = fmaf(a.x, b.x, fmaf(a.y, b.y, acc.x));
    acc.y = fmaf(a.x, b.y, fmaf(-a.y, b.x, acc.y));
}
LRCCS_DEV float2 shfl_xor2(float2 v, int m) {
    return make_float2(__shfl_xor_sync(0xffffffffu, v.x, m), __shfl_xor_sync(0xffffffffu, v.y, m));
}

// Upper-triangle pair enumeration of an r x r Hermitian matrix: p -> (a, b), a <= b.
LRCCS_DEV void pair_of(int p, int r, int &a, int &b) {
    int aa = 0;
    int rem = p;
    while (rem >= r - aa) { rem -= r - aa; ++aa; }
    a = aa;
    b = aa + rem;
}
LRCCS_DEV int pair_index(int a, int b, int r) {  // a <= b
    return a * r - (a * (a - 1)) / 2 + (b - a);
}

// |v|^2 in FP64 without contraction: the truncation decision |y|^2 <= gamma of
// the spectral initialisation is taken on exactly the squares an FP64
// reference forms.
LRCCS_DEV double abs2_rn(float2 v) {
    return __dadd_rn(__dmul_rn((double)v.x, (double)v.x), __dmul_rn((double)v.y, (double)v.y));
}

// |v|^2 > gam on those FP64 squares; the FP32 square decides wherever it is
// further from gam than its rounding (glo, ghi = gam (1 -+ 1e-5)) and in range
LRCCS_DEV bool trunc_drop(float2 v, double gam, float glo, float ghi) {
    if (v.x == 0.f && v.y == 0.f) return false;   // gam >= 0
    const float s = fmaf(v.x, v.x, v.y * v.y);
    if (s > 1e-30f && s < 1e30f) {
        if (s < glo) return false;
        if (s > ghi) return true;
    }
    return abs2_rn(v) > gam;
}

// Load the twiddle table of length N into shared memory.
LRCCS_DEV void load_twiddles(float2 *s_tw, const float2 *g_tw, int N) {
    for (int t = threadIdx.x; t < N; t += blockDim.x) s_tw[t] = g_tw[t];
}

// ---------------------------------------------------------------- grid reductions
//
// "Last block" pattern: each block writes its partial, fences, and increments a
// counter; the block that sees count == gridDim-1 reduces all partials in a
// fixed order (deterministic) and resets the counter for the next launch.
LRCCS_DEV bool last_block_arrive(unsigned int *counter) {
    __shared__ bool s_last;
    __threadfence();
    __syncthreads();
    if (threadIdx.x == 0) {
        unsigned int nblk = gridDim.x * gridDim.y * gridDim.z;
        unsigned int prev = atomicAdd(counter, 1u);
        s_last = (prev == nblk - 1);
        if (s_last) *counter = 0u;
    }
    __syncthreads();
    if (s_last) __threadfence();
    return s_last;
}

// ---------------------------------------------------------------- Hermitian eigensolver

// Parallel cyclic Jacobi for an n x n Hermitian matrix A in shared memory
// (all threads of the block call it).  Rounds follow the circle ordering, so
// the n/2 rotations of a round touch disjoint index pairs.  Each rotation
// removes the phase of a_pq and applies the real 2x2 Jacobi rotation:
// G = [[c, s], [-s e^{-i phi}, c e^{-i phi}]], A <- G^H A G, V <- V G.
// V (ldv columns, may be global memory) is updated when non-null.
// A rotation is skipped when |a_pq| <= rel_tol sqrt(|a_pp a_qq|) or |a_pq| <= abs_tol,
// or when both |a_pp| and |a_qq| are below tail_tol (a rotation between two
// such indices only mixes columns p and q of V: when every wanted eigenvalue
// is above tail_tol, the wanted eigenvectors converge without them);
// the sweeps stop when a whole sweep skips every rotation.
//
// One barrier a round: latency bounds a round, so the thread that rotates the
// 2 x 2 block holding a pivot of the next round forms that rotation from it at
// once (the pivot's two diagonal entries follow from the last round's and this
// round's t |a_pq|).  Only the blocks on and above the diagonal are rotated, the
// rest is their mirror image; other warps update V meanwhile.
// One matrix, first pass, whole-matrix rotations in two phases -> half blocks,
// rotations by one warp beside the V update -> this form: q = 32: 162 -> 145 ->
// 116 us, q = 48: 405 -> 269 -> 247, q = 64: 601 -> 429 -> 388,
// q = 96: 2040 -> 1173 -> 1006.
struct JacobiRot {
    float4 g[64];      // c, s, e
    float tb[64];      // t |a_pq|: a_pp falls by it, a_qq grows
    uint32_t pq[64];   // p | q << 16
};
struct JacobiWork {
    JacobiRot rot[2];
    float diag[2][128];   // the diagonal after an even / odd round
    int cnt[2];           // a sweep rotated something (by the sweep's parity)
};

// Rotation i of a round, of indices p and q; returns whether it is not skipped.
LRCCS_DEV bool jacobi_rotation(JacobiRot &r, int i, int p, int q, float2 apq, float al, float ga, float abs_tol,
                               float rel_tol, float tail_tol) {
    const float b2 = apq.x * apq.x + apq.y * apq.y;
    float c = 1.f, s = 0.f, tb = 0.f;
    float2 e = make_float2(1.f, 0.f);
    const bool live = b2 > 1e-36f && b2 > abs_tol * abs_tol &&
                      b2 > rel_tol * rel_tol * fabsf(al) * fabsf(ga) && (fabsf(al) >= tail_tol || fabsf(ga) >= tail_tol);
    if (live) {
        // the rotation only has to be orthogonal: c = 1 / sqrt(1 + t^2), s = t c
        // hold to rounding whatever the accuracy of t, so t takes the short forms
        // (tau^2 held finite); c is rounded to nearest: rsqrtf's bias took 1e-5
        // off V's column norms over 47 x 5 rotations, and off the singular values
        const float ib = rsqrtf(b2);
        e = make_float2(apq.x * ib, apq.y * ib);
        const float tau = (ga - al) * 0.5f * ib;
        const float h2 = fminf(fmaf(tau, tau, 1.f), 1e38f);
        const float t = __fdividef(copysignf(1.f, tau), fabsf(tau) + h2 * rsqrtf(h2));
        c = __frsqrt_rn(fmaf(t, t, 1.f));
        s = t * c;
        tb = t * (b2 * ib);
    }
    r.g[i] = make_float4(c, s, e.x, e.y);
    r.tb[i] = tb;
    r.pq[i] = p | q << 16;
    return live;
}

// Threads that hold blocks of A beside others that update V: one block each up
// to 17 warps (n = 64), then several; 1024 threads leave 15 warps for V.
__host__ __device__ inline int jacobi_block_threads(int n) {
    const int np = n > 5 ? (n + 1) / 2 : 3, t = (np * (np + 1) / 2 + 31) / 32 * 32;
    return t < 544 ? t : 544;
}

// PAD: A holds jacobi_rows(n) rows and columns, zero past n.
__host__ __device__ inline int jacobi_rows(int n) { return n > 5 ? n + (n & 1) : 6; }

template <bool PAD>
__device__ inline void block_jacobi(float2 *A, int n, int lda, float2 *V, int ldv, JacobiWork &w, int max_sweeps,
                                    float abs_tol = 0.f, float rel_tol = 1e-7f, float tail_tol = 0.f) {
    // at least three pairs (indices past n are never rotated): a block then holds at most one pivot
    const int n2 = jacobi_rows(n), npair = n2 / 2, nblk = npair * (npair + 1) / 2, N = n2 - 1;
    // This thread's blocks (i, i2), the same in every round: at most 2080 of them
    // (n <= 128), four a thread; the other warps update V.  Round rnd pairs
    // (rnd + i, rnd - i) mod N for i >= 1 and (rnd, N), so pivot x of the next round
    // lies in the rows of pair x - 1 and the columns of pair x + 1 (or at the ends
    // (0, 1) and (npair - 2, npair - 1)).  The pivots' blocks go to the first threads,
    // for few warps to run the rotations' code; the rest follow by rows.
    const int na = V ? jacobi_block_threads(n) : (int)blockDim.x;
    int blk[4];   // i << 8 | i2, -1: none
#pragma unroll
    for (int k = 0; k < 4; ++k) {
        const int task = threadIdx.x < na ? threadIdx.x + k * na : nblk;
        int i, i2;
        if (task < npair) {
            i = task == 0 ? 0 : task == npair - 1 ? npair - 2 : task - 1;
            i2 = task == 0 ? 1 : task == npair - 1 ? npair - 1 : task + 1;
        } else {
            int left = task - npair;
            for (i = 0; i < npair; ++i) {
                const bool e1 = i == 0 || i == npair - 2, e2 = i + 2 < npair;   // pivots at i + 1, i + 2
                const int cnt = npair - i - e1 - e2;
                if (left < cnt) {
                    i2 = i + left;
                    if (e1 && i2 >= i + 1) ++i2;
                    if (e2 && i2 >= i + 2) ++i2;
                    break;
                }
                left -= cnt;
            }
        }
        blk[k] = task < nblk ? i << 8 | i2 : -1;
    }
    const bool pivot = threadIdx.x < npair;   // blk[0] holds pivot threadIdx.x of the next round: its
    const bool prow = threadIdx.x != 1, pcol = threadIdx.x == npair - 1;   // second row, second column
    __syncthreads();
    if (threadIdx.x < 2) w.cnt[threadIdx.x] = 0;
    for (int i = threadIdx.x; i < n2; i += blockDim.x) w.diag[1][i] = i < n ? A[i * lda + i].x : 0.f;
    __syncthreads();
    for (int i = threadIdx.x; i < npair; i += blockDim.x) {
        const int p = i, q = i == 0 ? N : N - i;   // round 0
        const bool in = p < n && q < n;
        if (jacobi_rotation(w.rot[0], i, p, q, in ? A[p * lda + q] : make_float2(0.f, 0.f), w.diag[1][p],
                            w.diag[1][q], abs_tol, rel_tol, tail_tol))
            w.cnt[0] = 1;
    }
    __syncthreads();
    int b = 0;
    for (int sweep = 0; sweep < max_sweeps; ++sweep) {
        for (int rnd = 0; rnd < N; ++rnd, b ^= 1) {
            const JacobiRot &r = w.rot[b];
            const int nsweep = rnd == N - 1 ? sweep + 1 : sweep;   // the sweep of the next round
            if (rnd == 1 && threadIdx.x == 0) w.cnt[(sweep + 1) & 1] = 0;   // read by every thread before round 0
            // A <- G^H A G on the block (rows of pair i, columns of pair i2 >= i):
            // the row rotation first, then the column rotation
#pragma unroll
            for (int k = 0; k < 4; ++k) {
                if (blk[k] < 0) break;
                const int i = blk[k] >> 8, i2 = blk[k] & 255;
                const float4 g = r.g[i], g2 = r.g[i2];
                const bool turn = g.y != 0.f || g2.y != 0.f;
                if (!turn && !(k == 0 && pivot) && i != i2) continue;
                const uint32_t pq = r.pq[i], pq2 = r.pq[i2];
                const int p = pq & 0xffff, qq = pq >> 16, p2 = pq2 & 0xffff, q2 = pq2 >> 16;
                const bool r0 = PAD || p < n, r1 = PAD || qq < n, c0 = PAD || p2 < n, c1 = PAD || q2 < n;
                const float2 z = make_float2(0.f, 0.f);
                float2 a00 = r0 && c0 ? A[p * lda + p2] : z, a01 = r0 && c1 ? A[p * lda + q2] : z;
                float2 a10 = r1 && c0 ? A[qq * lda + p2] : z, a11 = r1 && c1 ? A[qq * lda + q2] : z;
                if (turn) {
                    // rows p, q of columns p2, q2 (the identity when skipped)
                    float c = g.x;
                    const float si = g.y, si2 = g2.y;
                    const float2 e = make_float2(g.z, g.w), eh = make_float2(g2.z, -g2.w);
                    float2 eaq = cmul(e, a10), ap = a00;
                    a00 = make_float2(c * ap.x - si * eaq.x, c * ap.y - si * eaq.y);
                    a10 = make_float2(si * ap.x + c * eaq.x, si * ap.y + c * eaq.y);
                    eaq = cmul(e, a11);
                    ap = a01;
                    a01 = make_float2(c * ap.x - si * eaq.x, c * ap.y - si * eaq.y);
                    a11 = make_float2(si * ap.x + c * eaq.x, si * ap.y + c * eaq.y);
                    // columns p2, q2 of rows p, q
                    c = g2.x;
                    float2 e2 = cmul(eh, a01);
                    ap = a00;
                    a00 = make_float2(c * ap.x - si2 * e2.x, c * ap.y - si2 * e2.y);
                    a01 = make_float2(si2 * ap.x + c * e2.x, si2 * ap.y + c * e2.y);
                    e2 = cmul(eh, a11);
                    ap = a10;
                    a10 = make_float2(c * ap.x - si2 * e2.x, c * ap.y - si2 * e2.y);
                    a11 = make_float2(si2 * ap.x + c * e2.x, si2 * ap.y + c * e2.y);
                }
                if (k == 0 && pivot) {   // (p', q') of the next round: column p', row q' of this block
                    const int pn = pcol ? q2 : p2, qn = prow ? qq : p;
                    const float *d = w.diag[b ^ 1];
                    const float al = d[pn] + (pcol ? r.tb[i2] : -r.tb[i2]), ga = d[qn] + (prow ? r.tb[i] : -r.tb[i]);
                    const float2 aqp = prow ? (pcol ? a11 : a10) : a00;
                    if (jacobi_rotation(w.rot[b ^ 1], threadIdx.x, pn, qn, cconj(aqp), al, ga, abs_tol, rel_tol,
                                        tail_tol))
                        w.cnt[nsweep & 1] = 1;
                }
                if (i2 == i) {
                    w.diag[b][p] = a00.x;
                    w.diag[b][qq] = a11.x;
                }
                if (!turn) continue;
                if (r0 && c0) A[p * lda + p2] = a00;
                if (r0 && c1) A[p * lda + q2] = a01;
                if (r1 && c0) A[qq * lda + p2] = a10;
                if (r1 && c1) A[qq * lda + q2] = a11;
                if (i2 != i) {   // the mirror block
                    if (r0 && c0) A[p2 * lda + p] = cconj(a00);
                    if (r0 && c1) A[q2 * lda + p] = cconj(a01);
                    if (r1 && c0) A[p2 * lda + qq] = cconj(a10);
                    if (r1 && c1) A[q2 * lda + qq] = cconj(a11);
                }
            }
            if (threadIdx.x >= na) {   // V <- V G: a warp takes columns p, q of pair i, a lane rows lane, lane + 32, ...
                const int nw = (blockDim.x - na) >> 5, lane = threadIdx.x & 31;
                for (int i = (threadIdx.x - na) >> 5; i < npair; i += nw) {
                    const float4 g = r.g[i];
                    const float c = g.x, s = g.y;
                    if (s == 0.f) continue;
                    const float2 eh = make_float2(g.z, -g.w);
                    float2 *vp = V + (r.pq[i] & 0xffff), *vq = V + (r.pq[i] >> 16);
#pragma unroll 2
                    for (int m = lane * ldv; m < n * ldv; m += 32 * ldv) {
                        const float2 a = vp[m], e2 = cmul(eh, vq[m]);
                        vp[m] = make_float2(c * a.x - s * e2.x, c * a.y - s * e2.y);
                        vq[m] = make_float2(s * a.x + c * e2.x, s * a.y + c * e2.y);
                    }
                }
            }
            __syncthreads();
        }
        if (w.cnt[sweep & 1] == 0) break;   // this sweep skipped every rotation
    }
    __syncthreads();
}

// Allow a kernel the device's opt-in shared memory per block, minus its static
// shared memory (the launch still requests only what it needs).
template <typename K>
static inline cudaError_t allow_smem(K kernel, int optin) {
    cudaFuncAttributes a;
    cudaError_t e = cudaFuncGetAttributes(&a, kernel);
    if (e != cudaSuccess) return e;
    return cudaFuncSetAttribute(kernel, cudaFuncAttributeMaxDynamicSharedMemorySize, optin - (int)a.sharedSizeBytes);
}

LRCCS_DEV double warp_sum_d(double v) {
#pragma unroll
    for (int o = 16; o > 0; o >>= 1) v += __shfl_xor_sync(0xffffffffu, v, o);
    return v;  // identical in every lane (each level adds the same two numbers)
}

// Compensated FP32 summation (Knuth's two-sum): a (hi, lo) pair carries ~48
// bits, at FP32 speed (an FP64 add is ~14x slower on this GPU).
struct fsum2 {
    float hi, lo;
};
LRCCS_DEV void two_sum(float a, float b, float &s, float &e) {
    s = a + b;
    const float bb = s - a;
    e = (a - (s - bb)) + (b - bb);
}
// FP32 sums of products without error: a product is the exact pair (p,
// fma(a, b, -p)), and p, its error term and the rounding of every addition go
// into three levels of two_sum (about 72 bits, more than an FP64 accumulator
// holds).  A product that leaves the FP32 range, or whose error term would (and
// NaN), goes to the FP64 sum `wide`.
struct fsum3 {
    float a, b, c;
};
LRCCS_DEV void fsum3_product(fsum3 &s, float a, float b) {   // 0 or 1e-26 <= |a b| <= 1e30
    const float p = __fmul_rn(a, b);
    float e, f;
    two_sum(s.a, p, s.a, e);
    two_sum(s.b, e, s.b, f);
    s.c += f;
    two_sum(s.b, fmaf(a, b, -p), s.b, f);
    s.c += f;
}
LRCCS_DEV void fsum3_mul(fsum3 &s, double &wide, float a, float b) {
    const float ap = fabsf(__fmul_rn(a, b));
    if (!(ap <= 1e30f && (ap >= 1e-26f || a == 0.f || b == 0.f))) {
        wide += (double)a * (double)b;
        return;
    }
    fsum3_product(s, a, b);
}
LRCCS_DEV double fsum3_total(const fsum3 &s) { return (double)s.a + ((double)s.b + (double)s.c); }
LRCCS_DEV void fsum_add(fsum2 &acc, float x) {
    float s, e;
    two_sum(acc.hi, x, s, e);
    acc.hi = s;
    acc.lo += e;
}
// Warp-wide sum of (hi, lo) pairs, kept as a pair; identical in every lane.
LRCCS_DEV fsum2 warp_fsum2(fsum2 v) {
#pragma unroll
    for (int o = 16; o > 0; o >>= 1) {
        const float oh = __shfl_xor_sync(0xffffffffu, v.hi, o), ol = __shfl_xor_sync(0xffffffffu, v.lo, o);
        float s, e;
        const bool first = (threadIdx.x & o) == 0;
        two_sum(first ? v.hi : oh, first ? oh : v.hi, s, e);
        v.lo = (first ? v.lo + ol : ol + v.lo) + e;
        v.hi = s;
    }
    return v;
}
// (hi, lo) pair sum a + b (a first)
LRCCS_DEV fsum2 fsum_pair(fsum2 a, fsum2 b) {
    float s, e;
    two_sum(a.hi, b.hi, s, e);
    fsum2 r;
    r.hi = s;
    r.lo = (a.lo + b.lo) + e;
    return r;
}
// Block-wide compensated sums dst[e] = sum_{m < nitem} fetch(e, m) for
// e < nent, written as FP64 (re, im) pairs.  Thread (entry e, slice s) sums
// items s, s + S, s + 2S, ... in that order with RB loads in flight, and the S
// slices are then combined by a fixed tree: deterministic, and one memory latency per
// RB items instead of one per item.  All threads of the block call it (the
// first 256 do the work); it ends with a barrier.
template <class F>
LRCCS_DEV void block_sum(int nent, int nitem, double *dst, F fetch) {
    constexpr int RB = 16;
    __shared__ float4 s_acc[256];   // (hi, lo) of re and im per thread
    const int nt = blockDim.x < 256 ? (int)blockDim.x : 256;
    const int t = threadIdx.x;
    const bool act = t < nt;   // threads beyond the first 256 only meet the barriers
    const int S = nent >= nt ? 1 : max(1, min(nt / nent, nitem));
    for (int base = 0; base < nent; base += nt) {
        const int e = base + (S == 1 ? t : t % nent), s = S == 1 ? 0 : t / nent;
        fsum2 re = {0.f, 0.f}, im = {0.f, 0.f};
        if (act && e < nent && s < S) {
            for (int m = s; m < nitem; m += S * RB) {
                float2 v[RB];
#pragma unroll
                for (int u = 0; u < RB; ++u) {
                    const int mm = m + u * S;
                    v[u] = mm < nitem ? fetch(e, mm) : make_float2(0.f, 0.f);
                }
#pragma unroll
                for (int u = 0; u < RB; ++u) {
                    fsum_add(re, v[u].x);
                    fsum_add(im, v[u].y);
                }
            }
        }
        if (S == 1) {
            if (act && e < nent) {
                dst[2 * e] = (double)re.hi + (double)re.lo;
                dst[2 * e + 1] = (double)im.hi + (double)im.lo;
            }
            continue;
        }
        // the slices add by a fixed tree (a thread per entry adding them one by
        // one waits for shared memory S times)
        if (act) s_acc[t] = make_float4(re.hi, re.lo, im.hi, im.lo);
        int h = 1;
        while (2 * h < S) h <<= 1;
        for (; h > 0; h >>= 1) {
            __syncthreads();
            if (act && e < nent && s < h && s + h < S) {
                const float4 b = s_acc[t + h * nent];
                re = fsum_pair(re, fsum2{b.x, b.y});
                im = fsum_pair(im, fsum2{b.z, b.w});
                s_acc[t] = make_float4(re.hi, re.lo, im.hi, im.lo);
            }
        }
        if (act && s == 0 && e < nent) {
            dst[2 * e] = (double)re.hi + (double)re.lo;
            dst[2 * e + 1] = (double)im.hi + (double)im.lo;
        }
    }
    __syncthreads();
}

// ---------------------------------------------------------------- grid barrier of a cooperative launch

// Barrier number k (1, 2, ...) of this launch: wait until every block has
// arrived k times (plus `skew` arrivals, which only the timeout test sets and
// the grid can never make).  Bounded: gives up after `limit` polls (2^24, 3.5
// seconds) and ORs `timeout_bit` into the status word; the kernel then runs on
// to its end.
LRCCS_DEV void grid_sync(unsigned int *bar, unsigned int k, unsigned int *status, unsigned int limit,
                         unsigned int skew, unsigned int timeout_bit) {
    __syncthreads();
    if (threadIdx.x == 0) {
        const unsigned int target = k * gridDim.x + skew;
        // the release covers the block's writes (ordered before it by the
        // barrier above), the acquire orders the others' before the one below
        asm volatile("red.release.gpu.global.add.u32 [%0], 1;\n" ::"l"(bar) : "memory");
        unsigned int v = 0, spins = 0;
        while (true) {
            asm volatile("ld.acquire.gpu.global.u32 %0, [%1];\n" : "=r"(v) : "l"(bar) : "memory");
            if (v >= target) break;
            if (++spins > limit) {
                atomicOr(status, timeout_bit);
                break;
            }
        }
    }
    __syncthreads();
}

// ---------------------------------------------------------------- asynchronous global -> shared copies
// cp.async keeps many copies in flight per thread without staging through
// registers; cp_async_wait() waits for all of this thread's copies, after
// which a __syncthreads() publishes the tile to the block.

LRCCS_DEV unsigned smem_u32(const void *p) { return (unsigned)__cvta_generic_to_shared(p); }

// 8-byte copy (one complex64); src must be 8-byte aligned.
LRCCS_DEV void cp_async8(void *dst, const void *src) {
    asm volatile("cp.async.ca.shared.global [%0], [%1], 8;\n" ::"r"(smem_u32(dst)), "l"(src) : "memory");
}
// 16-byte copy (two complex64); src and dst must be 16-byte aligned.
LRCCS_DEV void cp_async16(void *dst, const void *src) {
    asm volatile("cp.async.cg.shared.global [%0], [%1], 16;\n" ::"r"(smem_u32(dst)), "l"(src) : "memory");
}
// The same copies, or zeros (and no read) when !on.
LRCCS_DEV void cp_async8_or_zero(void *dst, const void *src, bool on) {
    asm volatile("cp.async.ca.shared.global [%0], [%1], 8, %2;\n" ::"r"(smem_u32(dst)), "l"(src), "r"(on ? 8 : 0)
                 : "memory");
}
LRCCS_DEV void cp_async16_or_zero(void *dst, const void *src, bool on) {
    asm volatile("cp.async.cg.shared.global [%0], [%1], 16, %2;\n" ::"r"(smem_u32(dst)), "l"(src), "r"(on ? 16 : 0)
                 : "memory");
}
// base + k strides of `bytes` bytes (one multiply-add with a constant k)
template <class V>
LRCCS_DEV V *step_by(V *base, unsigned bytes, unsigned k) {
    return (V *)((uintptr_t)base + (unsigned long long)bytes * k);
}
// A global store under a predicate: no branch around it.
LRCCS_DEV void st_global_if(float2 *p, float2 v, uint32_t on) {
    asm volatile("{\n.reg .pred p;\nsetp.ne.u32 p, %3, 0;\n@p st.global.v2.f32 [%0], {%1, %2};\n}\n" ::"l"(p), "f"(v.x),
                 "f"(v.y), "r"(on)
                 : "memory");
}
// Stage `count` complex64 values from global `src` into shared `dst`, 16 bytes
// per copy when both are 16-byte aligned and count is even, else 8 bytes.
LRCCS_DEV void stage_row(float2 *dst, const float2 *src, int count, int tid, int nthr) {
    if (((((uintptr_t)src) | smem_u32(dst)) & 15) == 0 && (count & 1) == 0) {
        for (int e = tid; e < count / 2; e += nthr) cp_async16(dst + 2 * e, src + 2 * e);
    } else {
        for (int e = tid; e < count; e += nthr) cp_async8(dst + e, src + e);
    }
}
LRCCS_DEV void cp_async_commit() { asm volatile("cp.async.commit_group;\n" ::: "memory"); }
LRCCS_DEV void cp_async_wait() { asm volatile("cp.async.wait_group 0;\n" ::: "memory"); }
// wait until at most one (two) committed groups are still pending
LRCCS_DEV void cp_async_wait_1() { asm volatile("cp.async.wait_group 1;\n" ::: "memory"); }
LRCCS_DEV void cp_async_wait_2() { asm volatile("cp.async.wait_group 2;\n" ::: "memory"); }

// ---------------------------------------------------------------- bulk copies (TMA)
// A bulk copy lands in shared memory and completes a transaction count on an
// mbarrier: one thread arms the barrier with the bytes and issues the copies,
// every thread waits on it.  The wait is bounded: false when it gave up.

LRCCS_DEV void mbar_init(uint64_t *bar, unsigned count) {
    asm volatile("mbarrier.init.shared::cta.b64 [%0], %1;\n" ::"r"(smem_u32(bar)), "r"(count) : "memory");
    asm volatile("fence.mbarrier_init.release.cluster;\n" ::: "memory");
}
LRCCS_DEV bool mbar_wait(uint64_t *bar, unsigned parity, unsigned limit) {
    unsigned done = 0;
    for (unsigned it = 0; it < limit && !done; ++it) {
        asm volatile(
            "{\n.reg .pred p;\nmbarrier.try_wait.parity.shared::cta.b64 p, [%1], %2;\nselp.u32 %0, 1, 0, p;\n}\n"
            : "=r"(done)
            : "r"(smem_u32(bar)), "r"(parity)
            : "memory");
    }
    return done != 0;
}
