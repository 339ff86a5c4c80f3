// Levenberg-Marquardt update on the device (Algorithm 1's Terminate() and
// f(), left to the minimiser by the paper, Sec. 2.2).
//
// One thread block per context.  After each fused evaluation at the trial
// offsets it (1) accepts the trial if chi^2 went down (lam /= 10, floored at
// lam_min) or rejects it (lam *= 10), (2) applies the stop rules, and (3) solves
// the damped system (H + lam diag(H)) delta = -g for the next trial, either
// over all 2 n_ant parameters (the full Gauss-Newton matrix: per-antenna 2x2
// diagonal blocks and one 2x2 cross block per baseline) or per antenna from
// the diagonal block alone with the step scaled by the loop gain block_gain.
// Parameters whose diagonal is not positive (antennas with no data) are held
// fixed.
//
// Precision.  GB300 runs FP64 at a small fraction of its FP32 rate, so the full
// system is factored in FP32 (Cholesky) and the solution is refined in FP64:
// the residual b - A x is formed in FP64 from the normal blocks themselves and
// the correction solved with the FP32 factor, until max|r| <= 1e-12 max|b| (at
// most 6 rounds).  That gives the FP64 solution for any matrix whose condition
// number is well below 1e7.  If the FP32 factorisation meets a non-positive
// pivot or the refinement does not converge, the system is assembled and
// factored in FP64 instead.
//
// Shape.  What costs here is not arithmetic (20 M multiply-adds for 197
// antennas) but serial chains, on one SM at that.  So as little as possible runs in
// sequence, and each refinement round is a product with an explicit inverse.
// Up to 2 n_ant = 90, one block inverts the matrix by Gauss-Jordan elimination in
// registers (6 x 6 elements a thread, one barrier a pivot).  Larger systems run on
// a cluster of eight blocks with the matrices in L2: one warp of each factors a
// 32 x 32 diagonal block in registers and inverts it (every block for itself,
// cheaper than waiting for it), the rows below are a product with that inverse,
// the trailing update goes in 64 x 64 tiles, and once L is complete W = L^-1 is
// formed by columns; a round is then y = W r, d += W^T y.
// Measured: 27 antennas 36 us a call (Cholesky column by column: 75; the
// cluster form on one block: 63), 197
// antennas 369 us (one block, solves from the factor: 1810).
#include <math.h>

#include <algorithm>

#include "psc_internal.cuh"

namespace psc {
namespace {

constexpr int kLmThreads = 256;
constexpr int kWarps = kLmThreads / 32;
constexpr int kSmallN2 = 90;            // 2 n_ant up to this: one block, matrices in shared memory
constexpr int kCluster = 8;             // blocks of a larger system
constexpr int kRefineMax = 6;
constexpr double kRefineTol = 1e-12;
constexpr int kPan = 32;                // panel width of the factorisation: one warp's lanes
constexpr int kTile = 64;               // trailing-update tile, 4 x 4 elements per thread
constexpr int kLd = kPan + 1;           // padded row of the shared tiles
constexpr unsigned kFull = 0xffffffffu;

__device__ __forceinline__ float warp_sum(float v) {
    for (int o = 16; o > 0; o >>= 1) v += __shfl_xor_sync(kFull, v, o);
    return v;
}

// Largest of the block's values, all >= 0 (whose bit patterns order as the
// values: the FP64 units are not asked).  A NaN counts as largest.
__device__ double block_max(double v, double *s) {
    long long m = __double_as_longlong(v);
    for (int o = 16; o > 0; o >>= 1) m = max(m, __shfl_xor_sync(kFull, m, o));
    __syncthreads();                                     // s may still be read from the last call
    if ((threadIdx.x & 31) == 0) s[threadIdx.x >> 5] = __longlong_as_double(m);
    __syncthreads();
    m = __double_as_longlong(s[0]);
    for (int w = 1; w < kWarps; ++w) m = max(m, __double_as_longlong(s[w]));
    return __longlong_as_double(m);
}

// Barrier of all threads that work on one system (a hardware barrier of the
// cluster, which orders their global writes and reads; or of the block).
template <bool kLarge>
__device__ __forceinline__ void sys_sync() {
    if constexpr (kLarge) asm volatile("barrier.cluster.arrive.release;\nbarrier.cluster.wait.acquire;" ::: "memory");
    else __syncthreads();
}

// What another block may have written is read past L1.
template <bool kLarge, class T>
__device__ __forceinline__ T ld(const T *p) {
    if constexpr (kLarge) return __ldcg(p);
    else return *p;
}

// Floats of the shared tiles: the diagonal block and its inverse, then the larger
// of the trailing update's two tiles and the inversion's rows of L and 16 columns of W.
__host__ __device__ inline size_t tile_floats(int n2) {
    const size_t wj = (size_t)kWarps * 4 * kPan + (size_t)(n2 + kPan - 1) / kPan * kPan * 16;
    const size_t tr = 2 * (size_t)kTile * kLd;
    return 2 * (size_t)kPan * kLd + (wj > tr ? wj : tr);
}

// The matrices and exchanged vectors of one system: shared memory (small) or
// the context's mat and mat32 (large).  Small systems keep A^-1 in place of A.
struct SysMem {
    float *A;          // [n2][n2] lower triangle of the damped matrix, then L below its diagonal blocks
    float *W;          // [n2][n2] lower triangle: L^-1
    float *y;          // [n2]
    double *r;         // [n2] residual
    double *d;         // [n2] solution
};

// Shared memory of one system's block.
struct SysShared {
    double *b, *r, *d;       // [n2] right-hand side, residual, solution
    float *r32, *y;          // [n2]
    int *ok;                 // [n2] the parameter has data (a positive diagonal)
    double *X;               // small systems: [n_bl][4] cross blocks, read by every residual
    float *ws;               // tiles: see lm_dyn_smem
};

// One warp: Cholesky of the 32 x 32 block D (lower triangle, row r in D[r kLd ..])
// in place and its inverse to I; lane r holds row r.  Returns nonzero if a pivot
// is not positive.
__device__ __forceinline__ int chol_diag(float *D, float *I) {
    const int lane = threadIdx.x & 31;
    float x[kPan];
    int bad = 0;
#pragma unroll
    for (int c = 0; c < kPan; ++c) x[c] = D[lane * kLd + c];
#pragma unroll
    for (int c = 0; c < kPan; ++c) {
        const float d = __shfl_sync(kFull, x[c], c);
        const bool nonpos = !(d > 0.f);
        bad |= nonpos;
        const float inv = nonpos ? 1.f : rsqrtf(d);
        x[c] *= inv;
#pragma unroll
        for (int t = c + 1; t < kPan; ++t) {
            const float l = __shfl_sync(kFull, x[c], t);
            x[t] = fmaf(-x[c], l, x[t]);
        }
        if (lane == c) I[c] = inv;                      // 1 / L_cc for the inverse, below
    }
    // the empty asm statements keep the compiler from merging these phases: where it
    // did, the function took 63 us instead of 5
    asm volatile("" ::: "memory");
    __syncwarp();
#pragma unroll
    for (int c = 0; c < kPan; ++c) D[lane * kLd + c] = x[c];
    float rd[kPan];
#pragma unroll
    for (int c = 0; c < kPan; ++c) rd[c] = I[c];
    __syncwarp();
    asm volatile("" ::: "memory");
    // column `lane` of the inverse: v_i = (delta - sum_{t<i} L_it v_t) / L_ii
    float v[kPan];
#pragma unroll
    for (int i = 0; i < kPan; ++i) {
        float s0 = i == lane ? 1.f : 0.f, s1 = 0.f;
#pragma unroll
        for (int t = 0; t < i; ++t) {
            if (t & 1) s1 = fmaf(-D[i * kLd + t], v[t], s1);
            else s0 = fmaf(-D[i * kLd + t], v[t], s0);
        }
        v[i] = (s0 + s1) * rd[i];
    }
    asm volatile("" ::: "memory");
    __syncwarp();
#pragma unroll
    for (int i = 0; i < kPan; ++i) I[i * kLd + lane] = v[i];
    __syncwarp();
    return bad;
}

// W = A^-1 (both triangles, rows of ldw) of a small system from A's lower triangle,
// by Gauss-Jordan elimination without pivoting (A is positive definite: its pivots
// are those of Cholesky's factorisation, squared).  Thread (tx, ty) holds elements
// (ty + 16 i, tx + 16 j); rc: 4 x 96 floats.  W may be A itself.  Returns nonzero
// (uniformly) if a pivot is not positive.
constexpr int kGj = (kSmallN2 + 15) / 16;
__device__ int gauss_jordan(const float *A, float *W, int ldw, int n, float *rc) {
    const int tx = threadIdx.x & 15, ty = threadIdx.x >> 4;
    float a[kGj][kGj];
#pragma unroll
    for (int i = 0; i < kGj; ++i)
#pragma unroll
        for (int j = 0; j < kGj; ++j) {
            const int r = ty + 16 * i, c = tx + 16 * j;
            a[i][j] = r < n && c < n ? A[(size_t)max(r, c) * n + min(r, c)] : (r == c ? 1.f : 0.f);
        }
    int bad = 0;
#pragma unroll
    for (int kb = 0; kb < kGj; ++kb) {
        const int k_hi = min(16, n - 16 * kb);
        for (int kk = 0; kk < k_hi; ++kk) {
            float *row = rc + (kk & 1) * 192, *col = row + 96;
            if (ty == kk) {
#pragma unroll
                for (int j = 0; j < kGj; ++j) row[tx + 16 * j] = a[kb][j];
            }
            if (tx == kk) {
#pragma unroll
                for (int i = 0; i < kGj; ++i) col[ty + 16 * i] = a[i][kb];
            }
            __syncthreads();
            const float p = row[16 * kb + kk];
            const bool nonpos = !(p > 0.f);
            bad |= nonpos;
            const float rp = nonpos ? 1.f : 1.f / p;
            float rj[kGj];
#pragma unroll
            for (int j = 0; j < kGj; ++j) rj[j] = row[tx + 16 * j] * rp;
            const bool my_row = ty == kk, my_col = tx == kk;
#pragma unroll
            for (int i = 0; i < kGj; ++i) {
                const float ci = col[ty + 16 * i];
#pragma unroll
                for (int j = 0; j < kGj; ++j) {
                    float v = fmaf(-ci, rj[j], a[i][j]);
                    if (j == kb && my_col) v = -ci * rp;
                    if (i == kb && my_row) v = j == kb && my_col ? rp : rj[j];
                    a[i][j] = v;
                }
            }
        }
        __syncthreads();                                 // an odd count would reuse the buffer still being read
    }
#pragma unroll
    for (int i = 0; i < kGj; ++i)
#pragma unroll
        for (int j = 0; j < kGj; ++j) {
            const int r = ty + 16 * i, c = tx + 16 * j;
            if (r < n && c < n) W[(size_t)r * ldw + c] = a[i][j];
        }
    __syncthreads();
    return bad;
}

// A = L L^T and W = L^-1 of one large system (see the file header).  Returns nonzero
// (uniformly) if a pivot is not positive.
__device__ int factor_invert(const SysMem &m, int n, float *ws, int rank, int nblk) {
    __shared__ int s_bad;
    const int tid = threadIdx.x, lane = tid & 31, warp = tid >> 5;
    const int tx = tid & 15, ty = tid >> 4;
    float *A = m.A, *W = m.W;
    float *D = ws, *I = ws + kPan * kLd;
    float *Ti = ws + 2 * kPan * kLd, *Tj = Ti + kTile * kLd;
    if (tid == 0) s_bad = 0;
    for (int k0 = 0; k0 < n; k0 += kPan) {
        const int kb = min(kPan, n - k0), m0 = k0 + kb;
        for (int e = tid; e < kPan * kPan; e += kLmThreads) {
            const int r = e / kPan, c = e % kPan;
            D[r * kLd + c] = (r < kb && c <= r) ? ld<true>(&A[(size_t)(k0 + r) * n + k0 + c]) : (r == c ? 1.f : 0.f);
        }
        __syncthreads();
        if (warp == 0) {
            const int bad = chol_diag(D, I);
            if (bad && lane == 0) s_bad = 1;
        }
        __syncthreads();
        if (rank == 0)
            for (int e = tid; e < kb * kPan; e += kLmThreads) {
                const int r = e / kPan, c = e % kPan;
                if (c < kb) W[(size_t)(k0 + r) * n + k0 + c] = I[r * kLd + c];
            }
        // rows below: L21 = A21 L11^-T, a warp per row (then the panel is full)
        if (m0 < n) {
            float li[kPan];
#pragma unroll
            for (int t = 0; t < kPan; ++t) li[t] = I[lane * kLd + t];
            const int step = nblk * kWarps;
            int i = m0 + rank * kWarps + warp;
            float a = i < n ? ld<true>(&A[(size_t)i * n + k0 + lane]) : 0.f;
            for (; i < n; i += step) {
                const float next = i + step < n ? ld<true>(&A[(size_t)(i + step) * n + k0 + lane]) : 0.f;
                float s0 = 0.f, s1 = 0.f;
#pragma unroll
                for (int t = 0; t < kPan; t += 2) {
                    s0 = fmaf(__shfl_sync(kFull, a, t), li[t], s0);
                    s1 = fmaf(__shfl_sync(kFull, a, t + 1), li[t + 1], s1);
                }
                A[(size_t)i * n + k0 + lane] = s0 + s1;
                a = next;
            }
        }
        sys_sync<true>();
        // trailing update: A22 -= L21 L21^T on the lower triangle, tile by tile
        const int nt = (n - m0 + kTile - 1) / kTile;
        int t = 0;
        for (int ti = 0; ti < nt; ++ti)
            for (int tj = 0; tj <= ti; ++tj, ++t) {
                if (t % nblk != rank) continue;
                const int i0 = m0 + ti * kTile, j0 = m0 + tj * kTile;
                for (int e = tid; e < kTile * kPan; e += kLmThreads) {
                    const int r = e / kPan, c = e % kPan;
                    Ti[r * kLd + c] = i0 + r < n ? ld<true>(&A[(size_t)(i0 + r) * n + k0 + c]) : 0.f;
                    Tj[r * kLd + c] = j0 + r < n ? ld<true>(&A[(size_t)(j0 + r) * n + k0 + c]) : 0.f;
                }
                float acc[4][4];
#pragma unroll
                for (int r = 0; r < 4; ++r) {
                    const int i = i0 + ty + 16 * r;
#pragma unroll
                    for (int c = 0; c < 4; ++c) {
                        const int j = j0 + tx + 16 * c;
                        acc[r][c] = i < n && j <= i ? ld<true>(&A[(size_t)i * n + j]) : 0.f;
                    }
                }
                __syncthreads();
#pragma unroll 8
                for (int q = 0; q < kPan; ++q) {
                    float li[4], lj[4];
#pragma unroll
                    for (int r = 0; r < 4; ++r) li[r] = Ti[(ty + 16 * r) * kLd + q];
#pragma unroll
                    for (int c = 0; c < 4; ++c) lj[c] = Tj[(tx + 16 * c) * kLd + q];
#pragma unroll
                    for (int r = 0; r < 4; ++r)
#pragma unroll
                        for (int c = 0; c < 4; ++c) acc[r][c] = fmaf(-li[r], lj[c], acc[r][c]);
                }
#pragma unroll
                for (int r = 0; r < 4; ++r) {
                    const int i = i0 + ty + 16 * r;
#pragma unroll
                    for (int c = 0; c < 4; ++c) {
                        const int j = j0 + tx + 16 * c;
                        if (i < n && j <= i) A[(size_t)i * n + j] = acc[r][c];
                    }
                }
                __syncthreads();
            }
        sys_sync<true>();
    }
    const int bad = s_bad;
    // W below its diagonal blocks: W_ij = -W_ii sum_{j <= k < i} L_ik W_kj, one block of
    // 16 columns at a time (the blocks shared out, longest first, forth and back); the
    // column block's rows so far stay in shared memory.  A warp takes four rows, lanes
    // (column, parity of k)
    float *Wj = ws + 2 * kPan * kLd + kWarps * 4 * kPan;     // [n][16], rows from 32 j
    float *Ls = ws + 2 * kPan * kLd + warp * 4 * kPan;       // the warp's four rows of L, [row][parity][16]
    float *S = D;
    const int nb = (n + kPan - 1) / kPan;
    const int col = lane & 15, par = lane >> 4, lpos = (lane & 1) * 16 + (lane >> 1);
    for (int u = 0; u < 2 * nb; ++u) {
        const int turn = u / nblk, at = u % nblk;
        if ((turn & 1 ? nblk - 1 - at : at) != rank) continue;
        const int j0 = (u >> 1) * kPan, cj = j0 + 16 * (u & 1);
        for (int e = tid; e < kPan * 16; e += kLmThreads) {
            const int r = e / 16, c = e % 16;
            Wj[e] = j0 + r < n && cj + c < n ? ld<true>(&W[(size_t)(j0 + r) * n + cj + c]) : 0.f;
        }
        __syncthreads();
        for (int i = (u >> 1) + 1; i < nb; ++i) {
            const int i0 = i * kPan, ib = min(kPan, n - i0);
            float acc[4] = {0.f, 0.f, 0.f, 0.f}, pre[4], wii[4];
#pragma unroll
            for (int r = 0; r < 4; ++r) {
                const int row = 4 * warp + r;
                pre[r] = row < ib ? ld<true>(&A[(size_t)(i0 + row) * n + j0 + lane]) : 0.f;
                wii[r] = row < ib && lane < ib ? ld<true>(&W[(size_t)(i0 + row) * n + i0 + lane]) : 0.f;
            }
            for (int k0 = j0; k0 < i0; k0 += kPan) {
                __syncwarp();
#pragma unroll
                for (int r = 0; r < 4; ++r) {
                    Ls[r * kPan + lpos] = pre[r];
                    if (k0 + kPan < i0 && 4 * warp + r < ib)
                        pre[r] = ld<true>(&A[(size_t)(i0 + 4 * warp + r) * n + k0 + kPan + lane]);
                }
                __syncwarp();
                const float *w = Wj + (k0 - j0) * 16 + lane;             // rows k0 + 2 q + par, column col
#pragma unroll
                for (int q = 0; q < 16; q += 4) {
                    const float w0 = w[q * 32], w1 = w[(q + 1) * 32], w2 = w[(q + 2) * 32], w3 = w[(q + 3) * 32];
#pragma unroll
                    for (int r = 0; r < 4; ++r) {
                        const float4 l = *reinterpret_cast<const float4 *>(Ls + r * kPan + par * 16 + q);
                        acc[r] = fmaf(l.x, w0, fmaf(l.y, w1, fmaf(l.z, w2, fmaf(l.w, w3, acc[r]))));
                    }
                }
            }
            __syncwarp();
#pragma unroll
            for (int r = 0; r < 4; ++r) {
                acc[r] += __shfl_xor_sync(kFull, acc[r], 16);
                if (par == 0) S[(4 * warp + r) * 16 + col] = acc[r];
                Ls[r * kPan + lpos] = wii[r];
            }
            __syncthreads();
#pragma unroll
            for (int r = 0; r < 4; ++r) {
                const int row = 4 * warp + r;
                float v = 0.f;
#pragma unroll
                for (int q = 0; q < 16; ++q) v = fmaf(-Ls[r * kPan + par * 16 + q], S[q * 32 + lane], v);
                v += __shfl_xor_sync(kFull, v, 16);
                if (par == 0) {
                    Wj[(i0 - j0 + row) * 16 + col] = v;
                    if (row < ib && cj + col < n) W[(size_t)(i0 + row) * n + cj + col] = v;
                }
            }
            __syncthreads();
        }
    }
    sys_sync<true>();
    return bad;
}

// The damped step of one system: (H + lam diag(H)) d = -g from src = chi2 | g |
// H | X.  On return sh.d holds it in every block; false if the FP32 factor or
// the refinement failed.
template <bool kLarge>
__device__ bool solve_damped(const LMArgs &a, const double *src, double lam, const SysMem &m, const SysShared &sh,
                             double *s_tmp, int rank, int nblk) {
    const int tid = threadIdx.x, lane = tid & 31, warp = tid >> 5;
    const int n = a.n_ant, n2 = 2 * n;
    const double *g = src + 1, *H = src + 1 + n2, *X = src + 1 + n2 + 3 * (size_t)n;
    // parameters without data (a diagonal that is not positive) are held fixed
    for (int p = tid; p < n2; p += kLmThreads) {
        sh.ok[p] = H[3 * (p >> 1) + ((p & 1) ? 2 : 0)] * (1.0 + lam) > 0.0;
        sh.b[p] = sh.ok[p] ? -g[p] : 0.0;
        sh.r[p] = sh.b[p];
    }
    __syncthreads();
    // FP32 lower triangle of the damped matrix
    for (int an = rank * kLmThreads + tid; an < n; an += nblk * kLmThreads) {
        const int p = 2 * an;
        const int o0 = sh.ok[p], o1 = sh.ok[p + 1];
        m.A[(size_t)p * n2 + p] = o0 ? (float)(H[3 * an] * (1.0 + lam)) : 1.f;
        m.A[(size_t)(p + 1) * n2 + p] = o0 && o1 ? (float)H[3 * an + 1] : 0.f;
        m.A[(size_t)(p + 1) * n2 + p + 1] = o1 ? (float)(H[3 * an + 2] * (1.0 + lam)) : 1.f;
    }
    for (int bl = rank * kLmThreads + tid; bl < a.n_bl; bl += nblk * kLmThreads) {
        const int2 ij = a.pairs[bl];
        const int p = 2 * ij.x, q = 2 * ij.y;           // i < j: the block (q, p) is below the diagonal
        const double *x = X + 4 * (size_t)bl;
        if constexpr (!kLarge) {
#pragma unroll
            for (int k = 0; k < 4; ++k) sh.X[4 * bl + k] = x[k];
        }
        const int pl = sh.ok[p], pm = sh.ok[p + 1], ql = sh.ok[q], qm = sh.ok[q + 1];
        float *r0 = m.A + (size_t)q * n2 + p, *r1 = r0 + n2;
        r0[0] = pl && ql ? (float)x[0] : 0.f;
        r1[0] = pl && qm ? (float)x[1] : 0.f;
        r0[1] = pm && ql ? (float)x[2] : 0.f;
        r1[1] = pm && qm ? (float)x[3] : 0.f;
    }
    sys_sync<kLarge>();
    if constexpr (kLarge) {
        if (factor_invert(m, n2, sh.ws, rank, nblk)) return false;
    } else {
        if (gauss_jordan(m.A, m.W, n2 + 1, n2, sh.ws)) return false;
    }
    double bmax = 0.0;
    for (int p = tid; p < n2; p += kLmThreads) bmax = fmax(bmax, fabs(sh.b[p]));
    bmax = block_max(bmax, s_tmp);
    float *red = sh.ws;                                  // [kWarps][32]
    for (int it = 0; it < kRefineMax; ++it) {
        for (int p = tid; p < n2; p += kLmThreads) sh.r32[p] = (float)sh.r[p];
        __syncthreads();
        if constexpr (!kLarge) {                             // d += A^-1 r, four lanes a row
            for (int p = tid >> 2; p < (n2 + 7) / 8 * 8; p += kLmThreads / 4) {
                float v = 0.f;
                if (p < n2)
                    for (int c = tid & 3; c < n2; c += 4) v = fmaf(m.W[(size_t)p * (n2 + 1) + c], sh.r32[c], v);
                v += __shfl_xor_sync(kFull, v, 1);
                v += __shfl_xor_sync(kFull, v, 2);
                if (p < n2 && (tid & 3) == 0) sh.d[p] = it == 0 ? (double)v : sh.d[p] + (double)v;
            }
            __syncthreads();
        } else {
            for (int p = rank * kWarps + warp; p < n2; p += nblk * kWarps) {       // y = W r
                const float *row = m.W + (size_t)p * n2;
                float s = 0.f;
                for (int c = lane; c <= p; c += 32) s = fmaf(ld<kLarge>(&row[c]), sh.r32[c], s);
                s = warp_sum(s);
                if (lane == 0) m.y[p] = s;
            }
            sys_sync<kLarge>();
            for (int p = tid; p < n2; p += kLmThreads) sh.y[p] = ld<kLarge>(&m.y[p]);
            __syncthreads();
            for (int c0 = 32 * rank; c0 < n2; c0 += 32 * nblk) {                   // d += W^T y, 32 columns at a time
                const int c = c0 + lane;
                float s = 0.f;
                if (c < n2) {
#pragma unroll 8
                    for (int p = c0 + warp; p < n2; p += kWarps)
                        s = fmaf(p >= c ? ld<kLarge>(&m.W[(size_t)p * n2 + c]) : 0.f, sh.y[p], s);
                }
                red[warp * 32 + lane] = s;
                __syncthreads();
                if (warp == 0 && c < n2) {
                    float v = 0.f;
                    for (int w = 0; w < kWarps; ++w) v += red[w * 32 + lane];
                    m.d[c] = it == 0 ? (double)v : m.d[c] + (double)v;
                }
                __syncthreads();
            }
            sys_sync<kLarge>();
            for (int p = tid; p < n2; p += kLmThreads) sh.d[p] = ld<kLarge>(&m.d[p]);
            __syncthreads();
        }
        // r = b - A d in FP64, eight lanes per antenna: a warp's FP64 instruction costs
        // the same for one lane as for 32, so few lanes may idle
        for (int a0 = (rank * kWarps + warp) * 4; a0 < n; a0 += nblk * kWarps * 4) {
            const int an = min(a0 + (lane >> 3), n - 1);
            double s0 = 0.0, s1 = 0.0;
#pragma unroll 2
            for (int o = lane & 7; o < n; o += 8) {
                if (o == an) continue;
                const double dl = sh.d[2 * o], dm = sh.d[2 * o + 1];      // zero where held
                const int i = min(an, o), j = max(an, o);
                const double *x = (kLarge ? X : sh.X) + 4 * ((size_t)i * (2 * n - i - 1) / 2 + (j - i - 1));
                const double xlm = an < o ? x[1] : x[2], xml = an < o ? x[2] : x[1];
                const int ol = sh.ok[2 * o], om = sh.ok[2 * o + 1];
                s0 = fma(ol ? x[0] : 0.0, dl, fma(om ? xlm : 0.0, dm, s0));
                s1 = fma(ol ? xml : 0.0, dl, fma(om ? x[3] : 0.0, dm, s1));
            }
#pragma unroll
            for (int o = 4; o > 0; o >>= 1) {
                s0 += __shfl_xor_sync(kFull, s0, o);
                s1 += __shfl_xor_sync(kFull, s1, o);
            }
            if ((lane & 7) == 0 && a0 + (lane >> 3) < n) {
                const int p = 2 * an, o0 = sh.ok[p], o1 = sh.ok[p + 1];
                const double dl = sh.d[p], dm = sh.d[p + 1], hlm = o0 && o1 ? H[3 * an + 1] : 0.0;
                s0 = fma(H[3 * an] * (1.0 + lam), dl, fma(hlm, dm, s0));
                s1 = fma(hlm, dl, fma(H[3 * an + 2] * (1.0 + lam), dm, s1));
                m.r[p] = o0 ? sh.b[p] - s0 : 0.0;
                m.r[p + 1] = o1 ? sh.b[p + 1] - s1 : 0.0;
            }
        }
        sys_sync<kLarge>();
        double rmax = 0.0;
        for (int p = tid; p < n2; p += kLmThreads) {
            sh.r[p] = ld<kLarge>(&m.r[p]);
            rmax = fmax(rmax, fabs(sh.r[p]));
        }
        rmax = block_max(rmax, s_tmp);
        if (rmax <= kRefineTol * bmax) return true;
    }
    sys_sync<kLarge>();                                  // the fallback writes over r, which others may still read
    return false;
}

// FP64 Cholesky + solve of A x = b in place (x overwrites b), all threads.
__device__ int chol64_solve(double *A, int n2, double *b) {
    __shared__ int s_bad;
    const int tid = threadIdx.x;
    if (tid == 0) s_bad = 0;
    __syncthreads();
    for (int k = 0; k < n2; ++k) {
        if (tid == 0) {
            const double d = A[(size_t)k * n2 + k];
            if (!(d > 0.0)) { s_bad = 1; A[(size_t)k * n2 + k] = 1.0; }
            else A[(size_t)k * n2 + k] = sqrt(d);
        }
        __syncthreads();
        const double lkk = A[(size_t)k * n2 + k];
        for (int i = k + 1 + tid; i < n2; i += blockDim.x) A[(size_t)i * n2 + k] /= lkk;
        __syncthreads();
        const int tx = tid & 15, ty = tid >> 4;
        for (int i = k + 1 + ty; i < n2; i += 16) {
            const double lik = A[(size_t)i * n2 + k];
            for (int j = k + 1 + tx; j <= i; j += 16) A[(size_t)i * n2 + j] -= lik * A[(size_t)j * n2 + k];
        }
        __syncthreads();
    }
    for (int k = 0; k < n2; ++k) {
        if (tid == 0) b[k] /= A[(size_t)k * n2 + k];
        __syncthreads();
        const double yk = b[k];
        for (int i = k + 1 + tid; i < n2; i += blockDim.x) b[i] -= A[(size_t)i * n2 + k] * yk;
        __syncthreads();
    }
    for (int k = n2 - 1; k >= 0; --k) {
        if (tid == 0) b[k] /= A[(size_t)k * n2 + k];
        __syncthreads();
        const double xk = b[k];
        for (int i = tid; i < k; i += blockDim.x) b[i] -= A[(size_t)k * n2 + i] * xk;
        __syncthreads();
    }
    return s_bad;
}

// FP64 matrix H + lam diag(H) (both triangles) and right-hand side -g, held parameters decoupled.
__device__ void assemble64(const LMArgs &a, const double *src, double lam, const int *ok, double *A, double *b) {
    const int tid = threadIdx.x, n = a.n_ant, n2 = 2 * n;
    const double *g = src + 1, *H = src + 1 + n2, *X = src + 1 + n2 + 3 * (size_t)n;
    for (int an = tid; an < n; an += kLmThreads) {
        const int p = 2 * an;
        const double hlm = ok[p] && ok[p + 1] ? H[3 * an + 1] : 0.0;
        A[(size_t)p * n2 + p] = ok[p] ? H[3 * an] * (1.0 + lam) : 1.0;
        A[(size_t)p * n2 + p + 1] = hlm;
        A[(size_t)(p + 1) * n2 + p] = hlm;
        A[(size_t)(p + 1) * n2 + p + 1] = ok[p + 1] ? H[3 * an + 2] * (1.0 + lam) : 1.0;
        b[p] = ok[p] ? -g[p] : 0.0;
        b[p + 1] = ok[p + 1] ? -g[p + 1] : 0.0;
    }
    for (int bl = tid; bl < a.n_bl; bl += kLmThreads) {
        const int2 ij = a.pairs[bl];
        for (int s = 0; s < 2; ++s)
            for (int t = 0; t < 2; ++t) {
                const int p = 2 * ij.x + s, q = 2 * ij.y + t;
                const double x = ok[p] && ok[q] ? X[4 * (size_t)bl + 2 * s + t] : 0.0;
                A[(size_t)p * n2 + q] = x;
                A[(size_t)q * n2 + p] = x;
            }
    }
    __syncthreads();
}

// One update; the blocks of a cluster (nblk, this one's rank) share a large
// system, block 0 alone takes a small one.  Every block comes to the same
// decisions from the same values.
template <bool kLarge>
__device__ void lm_update(const LMArgs &a, double *s_dyn, int rank, int nblk) {
    LMState *st = a.st;
    __shared__ double s_tmp[kLmThreads];
    const int tid = threadIdx.x;
    const int n = a.n_ant, n2 = 2 * n;
    const size_t len = ev_len(n, a.n_bl);
    const LMState s0 = *st;
    const double chi2_t = a.ev[0];                       // before the branch: one wait for both
    if (s0.done) return;

    // the step that produced this trial (its largest component)
    double tstep = 0.0;
    for (int p = tid; p < n2; p += kLmThreads) tstep = fmax(tstep, fabs(a.lm_trial[p] - a.lm_cur[p]));
    tstep = block_max(tstep, s_tmp);

    bool accept = false;
    int stop = PSC_STOP_NONE;
    double lam = s0.lam;
    if (s0.n_eval == 0) {
        if (isfinite(chi2_t)) accept = true;
        else stop = PSC_STOP_NUMERIC;
    } else if (isfinite(chi2_t) && chi2_t < s0.chi2) {
        accept = true;
        const double rel = s0.chi2 > 0.0 ? (s0.chi2 - chi2_t) / s0.chi2 : 0.0;
        lam = fmax(lam / 10.0, s0.lam_min);
        if (rel < s0.chi2_rtol) stop = PSC_STOP_CHI2;
    } else {
        lam *= 10.0;
        if (lam > s0.lam_max) stop = PSC_STOP_LAMBDA;
        // a rejected step already below ten times the step tolerance: the
        // minimum is found to within the evaluation's own noise, and a
        // rising lam would only shrink the step to the tolerance
        else if (isfinite(chi2_t) && tstep < 10.0 * s0.step_tol) stop = PSC_STOP_STEP;
    }
    if (stop == PSC_STOP_NONE && s0.n_iter >= s0.max_iter) stop = PSC_STOP_MAX_ITER;
    sys_sync<kLarge>();                                  // every block has read the state and the offsets
    if (rank == 0 && tid == 0) {
        st->n_eval = s0.n_eval + 1;
        if (accept) st->chi2 = chi2_t;
        st->lam = lam;
        if (stop != PSC_STOP_NONE) { st->reason = stop; st->done = 1; }
        else st->n_iter = s0.n_iter + 1;
    }
    if (accept) {
        for (size_t k = rank * kLmThreads + tid; k < len; k += nblk * kLmThreads) a.cur[k] = a.ev[k];
        if (rank == 0)
            for (int k = tid; k < n2; k += kLmThreads) a.lm_cur[k] = a.lm_trial[k];
    }
    if (stop != PSC_STOP_NONE) return;
    const double *src = accept ? a.ev : a.cur;           // cur is being written when it is the copy
    double *delta = a.rhs;
    bool fail = false;
    if (s0.mode == PSC_LM_BLOCK) {
        if (rank != 0) return;
        const double *g = src + 1, *H = src + 1 + n2;
        for (int an = tid; an < n; an += kLmThreads) {
            const double p = H[3 * an] * (1.0 + lam), b = H[3 * an + 1], d = H[3 * an + 2] * (1.0 + lam);
            const double det = p * d - b * b;
            double x0 = 0.0, x1 = 0.0;
            if (det > 0.0 && p > 0.0) {
                x0 = -(d * g[2 * an] - b * g[2 * an + 1]) / det;
                x1 = -(-b * g[2 * an] + p * g[2 * an + 1]) / det;
            }
            delta[2 * an] = s0.block_gain * x0;
            delta[2 * an + 1] = s0.block_gain * x1;
        }
        __syncthreads();
    } else {
        SysShared sh;
        sh.X = s_dyn;
        sh.b = s_dyn + (kLarge ? 0 : 4 * (size_t)a.n_bl);
        sh.r = sh.b + n2;
        sh.d = sh.r + n2;
        sh.r32 = (float *)(sh.d + n2);
        sh.y = sh.r32 + n2;
        sh.ok = (int *)(sh.y + n2);
        sh.ws = (float *)(sh.ok + n2);
        sh.ws += (4 - ((sh.ws - (float *)s_dyn) & 3)) & 3;                   // 16-byte aligned tiles
        SysMem m;
        if constexpr (kLarge) {
            m.d = a.rhs;
            m.A = a.mat32;
            m.W = (float *)a.mat;
            m.r = a.mat + ((size_t)n2 * n2 + 1) / 2;
            m.y = (float *)(m.r + n2);
        } else {
            m.A = sh.ws + 4 * 96;
            m.W = m.A;
            m.r = sh.r;
            m.y = sh.y;
            m.d = sh.d;
        }
        const bool solved = solve_damped<kLarge>(a, src, lam, m, sh, s_tmp, rank, nblk);
        if (rank != 0) return;
        if (solved) delta = sh.d;
        else {
            // FP64 fallback: factor the FP64 matrix itself
            assemble64(a, src, lam, sh.ok, a.mat, delta);
            fail = chol64_solve(a.mat, n2, delta) != 0;
            __syncthreads();
        }
    }

    double mx = 0.0;
    bool finite = true;
    for (int p = tid; p < n2; p += kLmThreads) {
        mx = fmax(mx, fabs(delta[p]));
        if (!isfinite(delta[p])) finite = false;
    }
    mx = block_max(finite ? mx : INFINITY, s_tmp);
    const bool numeric = fail || !isfinite(mx);
    if (numeric || mx < s0.step_tol) {
        if (tid == 0) { st->reason = numeric ? PSC_STOP_NUMERIC : PSC_STOP_STEP; st->done = 1; }
        return;
    }
    for (int p = tid; p < n2; p += kLmThreads) a.lm_trial[p] = a.lm_cur[p] + delta[p];
}

// Small systems, one block each.
__global__ void __launch_bounds__(kLmThreads) lm_small_kernel(const LMArgs a0, const LMArgs *__restrict__ la) {
    extern __shared__ __align__(16) double s_dyn[];
    const LMArgs a = la != nullptr ? la[blockIdx.x] : a0;
    lm_update<false>(a, s_dyn, 0, 1);
}

// Systems of any size, a cluster each (small ones in its first block).
__global__ void __launch_bounds__(kLmThreads) lm_cluster_kernel(const LMArgs a0, const LMArgs *__restrict__ la) {
    extern __shared__ __align__(16) double s_dyn[];
    const int rank = blockIdx.x % kCluster;
    const LMArgs a = la != nullptr ? la[blockIdx.x / kCluster] : a0;
    if (2 * a.n_ant <= kSmallN2) {
        if (rank == 0) lm_update<false>(a, s_dyn, 0, 1);
    } else {
        lm_update<true>(a, s_dyn, rank, kCluster);
    }
}

__global__ void lm_restart_kernel(const LMArgs a0, const LMState *st00, const double *lm00,
                                  const LMArgs *__restrict__ la, const LMState *const *st0s,
                                  const double *const *lm0s) {
    const bool batched = la != nullptr;
    const LMArgs a = batched ? la[blockIdx.x] : a0;
    const LMState *st0 = batched ? st0s[blockIdx.x] : st00;
    const double *lm0 = batched ? lm0s[blockIdx.x] : lm00;
    if (threadIdx.x == 0) *a.st = *st0;
    for (int p = threadIdx.x; p < 2 * a.n_ant; p += blockDim.x) {
        a.lm_trial[p] = lm0[p];
        a.lm_cur[p] = lm0[p];
    }
}

// Dynamic shared memory of the LM kernels: six vectors (b, r, d in FP64; r, y in
// FP32; the flags), then the tiles (large systems) or the pivot rows, the matrix (its
// inverse has rows of n2 + 1) and the cross blocks (small ones).
size_t lm_dyn_smem(int n_ant) {
    const int n2 = 2 * n_ant;
    const size_t n_bl = (size_t)n_ant * (n_ant - 1) / 2;
    const size_t base = (size_t)n2 * (3 * sizeof(double) + 2 * sizeof(float) + sizeof(int)) + 16;
    if (n2 <= kSmallN2) return base + sizeof(float) * (4 * 96 + (size_t)n2 * (n2 + 1)) + 4 * sizeof(double) * n_bl;
    return base + sizeof(float) * tile_floats(n2);
}

// Launches the update of n_ctx contexts: clusters if any of them is large.
cudaError_t launch_update(const LMArgs &a, const LMArgs *la, int n_ctx, size_t dyn, bool large, cudaStream_t s) {
    if (!large) {
        lm_small_kernel<<<n_ctx, kLmThreads, dyn, s>>>(a, la);
        return cudaGetLastError();
    }
    cudaLaunchConfig_t cfg{};
    cfg.gridDim = dim3(n_ctx * kCluster);
    cfg.blockDim = dim3(kLmThreads);
    cfg.dynamicSmemBytes = dyn;
    cfg.stream = s;
    cudaLaunchAttribute at[1];
    at[0].id = cudaLaunchAttributeClusterDimension;
    at[0].val.clusterDim.x = kCluster;
    at[0].val.clusterDim.y = at[0].val.clusterDim.z = 1;
    cfg.attrs = at;
    cfg.numAttrs = 1;
    return cudaLaunchKernelEx(&cfg, lm_cluster_kernel, a, la);
}

}  // namespace

cudaError_t lm_prepare(int n_ant) {
    (void)n_ant;
    const size_t most = std::max(lm_dyn_smem(kSmallN2 / 2), lm_dyn_smem(512));
    const cudaError_t e = cudaFuncSetAttribute(lm_small_kernel, cudaFuncAttributeMaxDynamicSharedMemorySize,
                                               (int)lm_dyn_smem(kSmallN2 / 2));
    if (e != cudaSuccess) return e;
    return cudaFuncSetAttribute(lm_cluster_kernel, cudaFuncAttributeMaxDynamicSharedMemorySize, (int)most);
}

size_t lm_smem_bytes(int n_ant) { return lm_dyn_smem(n_ant); }

cudaError_t launch_lm_restart(const LMArgs &a, const LMState *st0, const double *lm0, cudaStream_t s) {
    lm_restart_kernel<<<1, 128, 0, s>>>(a, st0, lm0, nullptr, nullptr, nullptr);
    return cudaGetLastError();
}

cudaError_t launch_lm_restart_batch(const LMArgs *la_dev, const LMState *const *st0_dev,
                                    const double *const *lm0_dev, int n_ctx, cudaStream_t s) {
    LMArgs none{};
    lm_restart_kernel<<<n_ctx, 128, 0, s>>>(none, nullptr, nullptr, la_dev, st0_dev, lm0_dev);
    return cudaGetLastError();
}

cudaError_t launch_lm_update(const LMArgs &a, cudaStream_t s) {
    return launch_update(a, nullptr, 1, lm_dyn_smem(a.n_ant), 2 * a.n_ant > kSmallN2, s);
}

cudaError_t launch_lm_update_batch(const LMArgs *la_dev, int n_ctx, size_t dyn, int max_ant, cudaStream_t s) {
    LMArgs none{};
    return launch_update(none, la_dev, n_ctx, dyn, 2 * max_ant > kSmallN2, s);
}

}  // namespace psc
