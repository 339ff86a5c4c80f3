// Fused evaluation kernel of the Pointing SelfCal hot path (sm_103a):
// degridding with the pointing-modified aperture kernel, the four pointing
// derivatives, the residual against the observed visibilities and the
// per-baseline sums of chi^2, gradient and Gauss-Newton normals.
//
// Paper basis (Bhatnagar & Cornwell 2017): Algorithm 1's inner loop; the
// kernel A_ij of Eq. AIJPOINTING and its derivative of Eq. DAIJPOINTING
// (extended to m, Sec. 3); chi^2 of Eq. Chisq and its gradient, Eq. DCHIDD.
//
// Work decomposition.  One thread block handles one "brick": a baseline
// (i, j), a group of c_group channels and t_tile * kv consecutive time steps.
// Each thread owns kv visibilities of one channel at consecutive times; they
// sit within a fraction of a grid cell of each other (the uv track moves
// slowly), so the thread walks the union of their tap rows and loads each
// grid cell once for all kv of them.  The block stages the grid cells its
// visibilities touch (the bounding box of their aperture disks) in shared
// memory.  The kernel's ramp factorises, exp(i pi (u_k - u_g) L) =
// exp(i pi (u_k - u_o) L) exp(-i pi (u_g - u_o) L) for any origin u_o, so the
// staged cells are pre-multiplied by the second factor (per cell, once per
// block) and each visibility applies the first factor once; the inner loop
// over taps then needs only the real radial A° and five FMAs per tap.  Taps
// outside the aperture's support are not visited, or read zero table entries
// (the tables are zero-padded far enough for every tap a thread visits).  If
// a brick's footprint does not fit the staging tile, the block falls back to
// reading the grid from global memory with the ramp applied per tap (same
// arithmetic, slower).
//
// Inner loop per tap and visibility (rho in units of table samples, t = rho
// ov): s2 = dxo^2 + dyo^2 (dxo = dx ov; dyo^2 carries a 1e-20 floor so s2 > 0),
// t = sqrt(s2) (hardware approximation, ~1 ulp), n = floor(t) by a round-toward-zero add of 2^23 whose bit
// pattern also gives the table address, A° = c_n + t s_n with the staged entry
// (c_n, s_n) = (A°(n) - n s_n, A°(n+1) - A°(n)) (the linear interpolation
// A°(n) + (t - n) s_n rearranged), then P += A° G', Q += (A° dxo) G' (each a
// packed FP32x2 FMA over the real and imaginary parts).
#include <algorithm>
#include <climits>

#include <cuda_bf16.h>

#include "psc_internal.cuh"
#include "tap_math.cuh"

namespace psc {
namespace {

using namespace tap;


// Grid cell (gy, gx) as FP32: from the bfloat16 copy when there is one
// (the widening is exact), else from the complex64 grid.
__device__ __forceinline__ float2 grid_cell(const EvalArgs &a, size_t idx) {
    if (a.grid_bf16 != nullptr) {
        const unsigned u = __ldg(&a.grid_bf16[idx]);
        return make_float2(__uint_as_float(u << 16), __uint_as_float(u & 0xFFFF0000u));
    }
    return __ldg(&a.grid[idx]);
}

// Shared memory of one block besides the dynamic tables; the staging tile only
// in instantiations that stage.
template <bool kTiled>
struct BlockSharedT {
    float2 tile[kTiled ? kTile * kTile : 1];
    float2 phx[kTile], phy[kTile];
    float red[kMaxThreads / 32][kRed];
    float red_c[kMaxThreads / 32][5];      // rounding errors of the compensated warp sums
    float bl[4];
    int box[4];
    int taps;          // taps of the brick's visibilities (pi rho_max^2 each, rounded up)
    int wp[2];         // residual-w stack: lowest and highest lower plane of the brick's visibilities
};

constexpr int kWCap = 3060;            // staged cells of all planes (24 KB: 4.85 ms in the case above; 32 KB 4.97, 40 KB 5.46, fewer blocks an SM)

// The tap sums of a rectangle's visibilities with a.split lanes per visibility:
// lane g takes rows g, g + split, ..., the row sums go through shared memory, and
// three of the lanes add them up in row order -- the additions of the one-lane loop
// in eval_brick, so every sum has the same bits.  For contexts with too few
// visibilities to fill the chip, where a lane's chain of some 600 taps is what the
// launch waits for: 21,060 visibilities, 185 us with a lane each, 56 us with 8.  A
// visibility's lanes sit in different warps: the lanes of one warp then walk the same
// row of neighbouring visibilities, spans of one length from neighbouring addresses
// (next to each other, in different rows, they took 70 us).  Shared memory s_split:
// [kMaxThreads] windows, [kMaxThreads][6] sums, then [support][kMaxThreads / split]
// row sums (P, Q).
__device__ __forceinline__ void split_taps(const EvalArgs &a, const float2 *s_tab, const BlockSharedT<true> &sh,
                                           float4 *s_split, int bl, int brick, int c_first, bool staged, int bx0, int by0) {
    const int tid = threadIdx.x, S = a.support;
    const int groups = blockDim.x / a.split, grp = tid & (groups - 1), sub = tid / groups;
    const int t_first = (brick % a.n_tt) * a.t_tile;
    const int n_t = min(a.t_tile, a.nt - t_first), n_c = min(a.c_group, a.nc - c_first);
    // an even number of cells a row and an aligned grid: every aligned pair of cells lies within it
    const bool pairs = a.grid_bf16 == nullptr && a.ng % 2 == 0 && ((uintptr_t)a.grid & 15) == 0;
    float *sums = reinterpret_cast<float *>(s_split + kMaxThreads);
    float4 *rows = s_split + kMaxThreads + kMaxThreads * 6 / 4 + grp;       // [support][groups]
    const float ov = (float)a.ov;
    for (int i0 = 0; i0 < n_t * n_c; i0 += groups) {
        const int i = i0 + grp;
        const bool on = i < n_t * n_c;
        const int lc = on ? i / n_t : 0, slot = on ? lc * a.t_tile + (i - lc * n_t) : 0;
        const float4 win = s_split[slot];
        const int ix0 = __float_as_int(win.x), iy0 = __float_as_int(win.y);
        const float hx = win.z, hy = win.w;
        const float rmax = a.chan[c_first + lc].rho_max, rmax2 = __fmul_rn(rmax, rmax);
        const unsigned tab_adj = (unsigned)__cvta_generic_to_shared(s_tab + lc * a.tab_stride) - (0x4B000000u << 3);
        int b_lo = max(0, (int)floorf(hy - rmax) + 1), b_hi = min(S - 1, (int)ceilf(hy + rmax) - 1);
        if (!staged) {
            b_lo = max(b_lo, -iy0);
            b_hi = min(b_hi, a.ng - 1 - iy0);
        }
        if (!on) b_hi = b_lo - 1;
        for (int b = b_lo + sub; b <= b_hi; b += a.split) {
            const float dy = hy - (float)b;
            const float dyo = dy * ov;
            const float dyo2 = fmaf(dyo, dyo, 1e-20f);
            const float rem = fmaf(-dy, dy, rmax2);      // written out, as are its factors: the span must not differ by a tap
            float2 P = make_float2(0.f, 0.f), Q = P;
            if (rem > 0.f) {
                const float r = fminf(rem * rsqrt_fast(rem), rmax);
                int a_lo = max(0, (int)floorf(hx - r) + 1), a_hi = min(S - 1, (int)ceilf(hx + r) - 1);
                if (staged) {
                    if (a_lo <= a_hi) {
                        float dxo[1] = {__fmul_rn(hx - (float)a_lo, ov)}, d2[1] = {dyo2};
                        float pr[1] = {0.f}, pi[1] = {0.f}, qr[1] = {0.f}, qi[1] = {0.f};
                        row_taps<1>(sh.tile + (iy0 - by0 + b) * kTile + (ix0 - bx0 + a_lo), a_hi - a_lo + 1, dxo, d2, ov,
                                    tab_adj, pr, pi, qr, qi);
                        P = make_float2(pr[0], pi[0]);
                        Q = make_float2(qr[0], qi[0]);
                    }
                } else {
                    a_lo = max(a_lo, -ix0);
                    a_hi = min(a_hi, a.ng - 1 - ix0);
                    float pr = 0.f, pi = 0.f, qr = 0.f, qi = 0.f;
                    if (a_lo <= a_hi) {
                        // Four cells at a time, the next four fetched ahead, as aligned pairs
                        // where rows hold them (one cell a load: 72 us); cells outside the
                        // row's span take a factor of zero, which leaves the sums.
                        const size_t row = (size_t)(iy0 + b) * a.ng + ix0;
                        const int first = pairs ? a_lo - ((ix0 + a_lo) & 1) : a_lo;
                        const int last = pairs ? a_hi - ((ix0 + a_hi) & 1) : a_hi;
                        auto load2 = [&](int aa) {
                            if (pairs) return __ldg(reinterpret_cast<const float4 *>(a.grid + row + min(aa, last)));
                            const float2 g0 = grid_cell(a, row + min(aa, last)), g1 = grid_cell(a, row + min(aa + 1, last));
                            return make_float4(g0.x, g0.y, g1.x, g1.y);
                        };
                        float dd = __fmul_rn(hx - (float)a_lo, ov);
                        float4 n0 = load2(first), n1 = load2(first + 2);
                        for (int aa = first; aa <= a_hi; aa += 4) {
                            const float2 gc[4] = {make_float2(n0.x, n0.y), make_float2(n0.z, n0.w),
                                                  make_float2(n1.x, n1.y), make_float2(n1.z, n1.w)};
                            n0 = load2(aa + 4);
                            n1 = load2(aa + 6);
#pragma unroll
                            for (int j = 0; j < 4; ++j) {
                                const bool in = aa + j >= a_lo && aa + j <= a_hi;
                                float2 g = cmul(gc[j], sh.phx[in ? aa + j : a_lo]);
                                g = make_float2(in ? g.x : 0.f, in ? g.y : 0.f);
                                const float d = in ? dd : 0.f;
                                const float s2 = fmaf(d, d, dyo2);
                                const float tv = sqrt_fast(s2);
                                const float tf = __fadd_rz(tv, 8388608.0f);
                                const float2 e = lds_f2(tab_adj + ((unsigned)__float_as_int(tf) << 3));
                                const float A = fmaf(tv, e.y, e.x);
                                pr = fmaf(A, g.x, pr);
                                pi = fmaf(A, g.y, pi);
                                const float Ad = __fmul_rn(A, d);
                                qr = fmaf(Ad, g.x, qr);
                                qi = fmaf(Ad, g.y, qi);
                                dd = in ? __fsub_rn(dd, ov) : dd;
                            }
                        }
                    }
                    const float2 py = sh.phy[b];
                    P = cmul(make_float2(pr, pi), py);
                    Q = cmul(make_float2(qr, qi), py);
                }
            }
            rows[b * groups] = make_float4(P.x, P.y, Q.x, Q.y);
        }
        __syncthreads();
        if (on && sub < 3) {
            // the first lane: sum P, the second: sum Q, the third: sum dy P, in row order
            float x = 0.f, y = 0.f;
            for (int b = b_lo; b <= b_hi; ++b) {
                const float2 v = reinterpret_cast<const float2 *>(rows + b * groups)[sub == 1];
                const float dy = hy - (float)b;
                x = sub == 2 ? fmaf(dy, v.x, x) : x + v.x;
                y = sub == 2 ? fmaf(dy, v.y, y) : y + v.y;
            }
            sums[6 * slot + 2 * sub] = x;
            sums[6 * slot + 2 * sub + 1] = y;
        }
        __syncthreads();
    }
}

// One brick: kv visibilities per thread.  acc receives the thread's 15 sums
// (reduce mode); predict mode writes V and the derivative planes.
// kW: the grid is a residual-w stack (EvalArgs::wp_n); every tap reads the two
// planes around its visibility's w and interpolates.  A brick's w changes slowly: the
// block stages the box of every plane that its visibilities touch (s_wtile, up to
// kWCap cells in all); bricks that need more read the planes tap by tap.  27 antennas, 600 x 64, 33 planes: 4.85 ms
// against 5.83 with every tap unstaged.
// kSplit: the rows of each visibility are shared among a.split lanes (split_taps);
// the brick, its sums and their order are those of the rectangle without it.
template <bool kPredict, int kV, bool kW, bool kSplit>
__device__ __forceinline__ void eval_brick(const EvalArgs &a, int brick, float2 *s_tab, BlockSharedT<!kW> &sh,
                                           float4 *s_split, float2 *s_wtile, float (&acc)[kRed], bool &active) {
    const int tid = threadIdx.x;
    // brick -> baseline, this thread's channel c and first time step t0, and
    // the block's channels [c_first, c_first + n_ch) (lc = c - c_first)
    int bl, c, t0, c_first, n_ch;
    if (a.flat > 0) {
        bl = brick / a.bpb;
        const int first = (brick - bl * a.bpb) * a.flat;
        const int k = first + tid;
        c = k / a.n_tp;
        t0 = (k - c * a.n_tp) * kV;
        c_first = first / a.n_tp;
        n_ch = min(a.nc - 1, (first + a.flat - 1) / a.n_tp) - c_first + 1;
        active = tid < a.flat && c < a.nc;
    } else {
        const int tt = brick % a.n_tt;
        const int cgi = (brick / a.n_tt) % a.n_cg;
        bl = brick / (a.n_tt * a.n_cg);
        const int lt = tid % a.t_tile;
        const int lcg = tid / a.t_tile;
        t0 = (tt * a.t_tile + lt) * kV;
        c_first = cgi * a.c_group;
        c = c_first + lcg;
        n_ch = a.c_group;
        active = lcg < a.c_group && t0 < a.nt && c < a.nc;
    }
    const int lc = c - c_first;
    const int tab_stride = a.tab_stride;
    const int S = a.support;

    // per-baseline constants, computed once per block in FP64
    if (tid == 0) {
        const int2 ij = a.pairs[bl];
        const double li = a.lm[2 * ij.x], mi = a.lm[2 * ij.x + 1];
        const double lj = a.lm[2 * ij.y], mj = a.lm[2 * ij.y + 1];
        sh.bl[0] = (float)(li + lj);   // ramp: l_i + l_j
        sh.bl[1] = (float)(mi + mj);
        sh.bl[2] = (float)(li - lj);   // decorrelation: l_i - l_j
        sh.bl[3] = (float)(mi - mj);
        sh.box[0] = INT_MAX; sh.box[1] = INT_MIN; sh.box[2] = INT_MAX; sh.box[3] = INT_MIN;
        sh.taps = 0;
        sh.wp[0] = INT_MAX; sh.wp[1] = INT_MIN;
    }
    __syncthreads();
    const float L = sh.bl[0], M = sh.bl[1], dL = sh.bl[2], dM = sh.bl[3];

    // Grid position of each visibility: x = u / du + Ng/2 (cells), window
    // origin floor(x) - S/2 + 1, hx = x - origin.  Times past the end of the
    // interval repeat the last one (computed, never stored), so every tap the
    // thread visits stays within its table padding.
    int ix0[kV], iy0[kV];
    float hx[kV], hy[kV];
    float rmax = 0.f;
    int wpl[kV];                                      // kW: the lower plane
    float wf[kV];                                     // kW: weight of the upper plane
    if (active) {
        const ChanConst ch = a.chan[c];
        rmax = ch.rho_max;
        int lox = INT_MAX, hix = INT_MIN, loy = INT_MAX, hiy = INT_MIN;
#pragma unroll
        for (int v = 0; v < kV; ++v) {
            const int t = min(t0 + v, a.nt - 1);
            int nx, ny;
            float fx, fy;
            if (a.uvs != nullptr) {
                const float4 q = a.uvs[(size_t)t * a.n_bl + bl];
                const float half = 0.5f * (float)a.ng;
                grid_pos(q.x, q.y, ch.sc_hi, ch.sc_lo, half, nx, fx);
                grid_pos(q.z, q.w, ch.sc_hi, ch.sc_lo, half, ny, fy);
            } else {
                const double *p = a.uvw + ((size_t)t * a.n_bl + bl) * 3;
                const double x = p[0] * ch.uv_scale + 0.5 * a.ng;
                const double y = p[1] * ch.uv_scale + 0.5 * a.ng;
                const double flx = floor(x), fly = floor(y);
                nx = (int)flx;
                ny = (int)fly;
                fx = (float)(x - flx);
                fy = (float)(y - fly);
            }
            if constexpr (kW) {
                const double *p = a.uvw + ((size_t)t * a.n_bl + bl) * 3;
                double q = (p[2] - a.wp_a * p[0] - a.wp_b * p[1]) * ch.uv_scale * a.wp_scale - a.wp_q0;
                q = fmin(fmax(q, 0.0), (double)(a.wp_n - 1));
                const int pl = min((int)floor(q), a.wp_n - 2);
                wpl[v] = pl;
                wf[v] = (float)(q - (double)pl);
            }
            ix0[v] = nx - S / 2 + 1;
            iy0[v] = ny - S / 2 + 1;
            hx[v] = fx + (float)(S / 2 - 1);
            hy[v] = fy + (float)(S / 2 - 1);
            // cells within rho_max of the visibility, inside its window
            lox = min(lox, ix0[v] + max(0, (int)floorf(hx[v] - rmax) + 1));
            hix = max(hix, ix0[v] + min(S - 1, (int)ceilf(hx[v] + rmax) - 1));
            loy = min(loy, iy0[v] + max(0, (int)floorf(hy[v] - rmax) + 1));
            hiy = max(hiy, iy0[v] + min(S - 1, (int)ceilf(hy[v] + rmax) - 1));
        }
        if (lox <= hix && loy <= hiy) {
            atomicMin(&sh.box[0], lox); atomicMax(&sh.box[1], hix);
            atomicMin(&sh.box[2], loy); atomicMax(&sh.box[3], hiy);
            const int nv = min(kV, a.nt - t0);
            atomicAdd(&sh.taps, nv * (int)ceilf(3.14159265f * rmax * rmax));
            if constexpr (kW) {
#pragma unroll
                for (int v = 0; v < kV; ++v) {
                    atomicMin(&sh.wp[0], wpl[v]);
                    atomicMax(&sh.wp[1], wpl[v]);
                }
            }
        }
    }
    // radial tables of this block's channels as (c_n, s_n), zero-padded
    for (int j = 0; j < (kSplit ? min(n_ch, a.nc - c_first) : n_ch); ++j) {
        const int cc = c_first + j;
        const int off = cc < a.nc ? a.chan[cc].tab_off : 0;
        const int len = cc < a.nc ? a.chan[cc].tab_len : 0;
        for (int n = tid; n < tab_stride; n += blockDim.x) {
            float2 v = make_float2(0.f, 0.f);
            if (n < len) {
                const float2 e = a.tabs[off + n];
                v = make_float2(fmaf(-(float)n, e.y, e.x), e.y);
            }
            s_tab[j * tab_stride + n] = v;
        }
    }
    __syncthreads();
    const bool empty = sh.box[0] > sh.box[1];         // no visibility of the brick has a tap
    const int bx0 = empty ? 0 : sh.box[0], by0 = empty ? 0 : sh.box[2];
    const int ex = empty ? 0 : sh.box[1] - bx0 + 1, ey = empty ? 0 : sh.box[3] - by0 + 1;
    // Staging pays when the brick's taps reuse its cells: a staged cell costs
    // a global load, two complex products and a store (about four unstaged
    // taps' extra work), so stage only boxes of at most taps / 4 cells that
    // fit the tile.  Uniform over the block.
    const int n_pl = kW && !empty ? sh.wp[1] - sh.wp[0] + 2 : 1;        // planes that the brick touches
    const bool staged = kW ? !a.no_stage && !empty && ex <= kTile && ey <= kTile && n_pl <= kWCap / (ex * ey) &&
                                 2 * n_pl * ex * ey <= sh.taps
                           : !a.no_stage && ex <= kTile && ey <= kTile && 4 * ex * ey <= sh.taps;

    // per-cell half of the ramp, exp(-i pi du (k_x L + k_y M)) = phx[k_x] phy[k_y],
    // with (k_x, k_y) relative to the tile origin (staged) or to each
    // visibility's window origin (unstaged: k < S)
    if (!empty) {
        const int nx = staged ? ex : S, ny = staged ? ey : S;
        for (int k = tid; k < nx; k += blockDim.x) {
            float s, co;
            sincospif(-(float)k * a.du * L, &s, &co);
            sh.phx[k] = make_float2(co, s);
        }
        for (int k = tid; k < ny; k += blockDim.x) {
            float s, co;
            sincospif(-(float)k * a.du * M, &s, &co);
            sh.phy[k] = make_float2(co, s);
        }
        __syncthreads();
    }
    if (!kW && staged && !empty) {
        // threads -> (column, row group) with shifts: 64 columns per pass for
        // blocks of >= 64 threads, 32 for a 32-thread block (two passes);
        // the row step blockDim >> cshift is >= 1 for every allowed block size
        const int cshift = blockDim.x >= kTile ? 6 : 5;
        const int cols = 1 << cshift;
        const int rstep = blockDim.x >> cshift;
        for (int xx = tid & (cols - 1); xx < ex; xx += cols) {
            const int gx = bx0 + xx;
            const bool xin = gx >= 0 && gx < a.ng;
            const float2 px = sh.phx[xx];
            for (int yy = tid >> cshift; yy < ey; yy += rstep) {
                const int gy = by0 + yy;
                float2 g = make_float2(0.f, 0.f);
                if (xin && gy >= 0 && gy < a.ng) g = grid_cell(a, (size_t)gy * a.ng + gx);
                sh.tile[yy * kTile + xx] = cmul(g, cmul(px, sh.phy[yy]));
            }
        }
        __syncthreads();
    }

    // ---- per-visibility tap sums (relative to each visibility's window) ----
    float2 S0[kV], Su[kV], Sv[kV];
#pragma unroll
    for (int v = 0; v < kV; ++v) S0[v] = Su[v] = Sv[v] = make_float2(0.f, 0.f);
    if (kW && staged) {
        const int p0 = sh.wp[0], cells = ex * ey;
        for (int k = tid; k < cells; k += blockDim.x) {
            const int yy = k / ex, xx = k - yy * ex;
            const int gx = bx0 + xx, gy = by0 + yy;
            const bool in = gx >= 0 && gx < a.ng && gy >= 0 && gy < a.ng;
            const float2 z = cmul(sh.phx[xx], sh.phy[yy]);
            const float2 *src = a.grid + (size_t)p0 * a.ng * a.ng + (in ? (size_t)gy * a.ng + gx : 0);
#pragma unroll 4
            for (int p = 0; p < n_pl; ++p, src += (size_t)a.ng * a.ng)
                s_wtile[p * cells + k] = in ? cmul(__ldg(src), z) : make_float2(0.f, 0.f);
        }
        __syncthreads();
        if (active) {
            const unsigned tab_adj = (unsigned)__cvta_generic_to_shared(s_tab + lc * tab_stride) - (0x4B000000u << 3);
            const float ov = (float)a.ov;
            const float rmax2 = rmax * rmax;
            int wx[kV], wy[kV];
            int r_lo = INT_MAX, r_hi = INT_MIN;
#pragma unroll
            for (int v = 0; v < kV; ++v) {
                wx[v] = ix0[v] - bx0;
                wy[v] = iy0[v] - by0;
                r_lo = min(r_lo, wy[v] + max(0, (int)floorf(hy[v] - rmax) + 1));
                r_hi = max(r_hi, wy[v] + min(S - 1, (int)ceilf(hy[v] + rmax) - 1));
            }
            for (int cy = r_lo; cy <= r_hi; ++cy) {
                float dy[kV], dyo2[kV];
                int c_lo = INT_MAX, c_hi = INT_MIN;
#pragma unroll
                for (int v = 0; v < kV; ++v) {
                    dy[v] = hy[v] - (float)(cy - wy[v]);
                    const float dyo = dy[v] * ov;
                    dyo2[v] = fmaf(dyo, dyo, 1e-20f);
                    const float rem = rmax2 - dy[v] * dy[v];
                    if (rem > 0.f) {
                        const float r = fminf(rem * rsqrt_fast(rem), rmax);
                        const int a_lo = max(0, (int)floorf(hx[v] - r) + 1);
                        const int a_hi = min(S - 1, (int)ceilf(hx[v] + r) - 1);
                        if (a_lo <= a_hi) {
                            c_lo = min(c_lo, wx[v] + a_lo);
                            c_hi = max(c_hi, wx[v] + a_hi);
                        }
                    }
                }
                if (c_lo > c_hi) continue;
                float dxo[kV], pr[kV], pi[kV], qr[kV], qi[kV];
#pragma unroll
                for (int v = 0; v < kV; ++v) {
                    dxo[v] = (hx[v] - (float)(c_lo - wx[v])) * ov;
                    pr[v] = pi[v] = qr[v] = qi[v] = 0.f;
                }
                const float2 *lo[kV];
#pragma unroll
                for (int v = 0; v < kV; ++v) lo[v] = s_wtile + (wpl[v] - p0) * cells + cy * ex + c_lo;
                row_taps_w<kV>(lo, cells, c_hi - c_lo + 1, dxo, dyo2, wf, ov, tab_adj, pr, pi, qr, qi);
#pragma unroll
                for (int v = 0; v < kV; ++v) {
                    S0[v].x += pr[v]; S0[v].y += pi[v];
                    Su[v].x += qr[v]; Su[v].y += qi[v];
                    Sv[v].x = fmaf(dy[v], pr[v], Sv[v].x);
                    Sv[v].y = fmaf(dy[v], pi[v], Sv[v].y);
                }
            }
        }
        const float inv_ov = 1.0f / (float)a.ov;
#pragma unroll
        for (int v = 0; v < kV; ++v) {                       // Q was accumulated with dx * ov
            Su[v].x *= inv_ov; Su[v].y *= inv_ov;
        }
    } else if constexpr (kSplit) {
        // each rectangle slot's window, then its sums in the same place
        if (active) s_split[tid] = make_float4(__int_as_float(ix0[0]), __int_as_float(iy0[0]), hx[0], hy[0]);
        __syncthreads();
        if (!empty) split_taps(a, s_tab, sh, s_split, bl, brick, c_first, staged, bx0, by0);
        __syncthreads();
        if (active && !empty) {
            const float *r = reinterpret_cast<const float *>(s_split + kMaxThreads) + 6 * tid;
            S0[0] = make_float2(r[0], r[1]);
            Su[0] = make_float2(r[2], r[3]);
            Sv[0] = make_float2(r[4], r[5]);
            const float inv_ov = 1.0f / (float)a.ov;
            Su[0].x *= inv_ov; Su[0].y *= inv_ov;
        }
    } else if (active && !empty) {
        const float2 *tab = s_tab + lc * tab_stride;
        const unsigned tab_adj = (unsigned)__cvta_generic_to_shared(tab) - (0x4B000000u << 3);
        const float ov = (float)a.ov;
        // the taps' operations are written out (here, in split_taps and row_taps): contracted
        // another way, a span may gain or lose a tap at its edge, a tap its offset's last bit
        const float rmax2 = __fmul_rn(rmax, rmax);
        if (!kW && staged) {
            int wx[kV], wy[kV];
            int r_lo = INT_MAX, r_hi = INT_MIN;
#pragma unroll
            for (int v = 0; v < kV; ++v) {
                wx[v] = ix0[v] - bx0;
                wy[v] = iy0[v] - by0;
                r_lo = min(r_lo, wy[v] + max(0, (int)floorf(hy[v] - rmax) + 1));
                r_hi = max(r_hi, wy[v] + min(S - 1, (int)ceilf(hy[v] + rmax) - 1));
            }
            if constexpr (kV == 2) {
                // two rows at a time over the wider one's columns (the one nearer the
                // centre's): the taps this adds read zero entries (at most rho_max + spread
                // + 1 cells away), as do those of a row past the last (whose cells are the
                // last row's again).  27 antennas, 150 x 64: 785 us an evaluation and 723 us
                // a prediction with derivatives against 813 and 775 a row at a time
                const float2 ov2 = make_float2(ov, ov), eps2 = make_float2(1e-20f, 1e-20f);
                for (int cy = r_lo; cy <= r_hi; cy += 2) {
                    const float2 dya = make_float2(hy[0] - (float)(cy - wy[0]), hy[1] - (float)(cy - wy[1]));
                    const float2 dyb = fadd2(dya, make_float2(-1.f, -1.f));
                    int c_lo = INT_MAX, c_hi = INT_MIN;
#pragma unroll
                    for (int v = 0; v < 2; ++v) {
                        const float da = v ? dya.y : dya.x;
                        const float d = fminf(fabsf(da), fabsf(da - 1.f));
                        const float rem = rmax2 - d * d;
                        if (rem > 0.f) {
                            // r <= rho_max keeps the span inside the staged box
                            const float r = fminf(rem * rsqrt_fast(rem), rmax);
                            c_lo = min(c_lo, wx[v] + max(0, (int)floorf(hx[v] - r) + 1));
                            c_hi = max(c_hi, wx[v] + min(S - 1, (int)ceilf(hx[v] + r) - 1));
                        }
                    }
                    if (c_lo > c_hi) continue;
                    const float2 dxo = make_float2((hx[0] - (float)(c_lo - wx[0])) * ov, (hx[1] - (float)(c_lo - wx[1])) * ov);
                    const float2 oa = fmul2(dya, ov2), ob = fmul2(dyb, ov2);
                    const float2 *row = sh.tile + cy * kTile + c_lo;
                    float2 pa[2], pb[2], q[2];
                    row_pair_taps2(row, cy < r_hi ? row + kTile : row, c_hi - c_lo + 1, dxo, ffma2(oa, oa, eps2),
                                   ffma2(ob, ob, eps2), ov, tab_adj, pa, pb, q);
#pragma unroll
                    for (int v = 0; v < 2; ++v) {
                        const float da = v ? dya.y : dya.x, db = v ? dyb.y : dyb.x;
                        S0[v].x += pa[v].x + pb[v].x; S0[v].y += pa[v].y + pb[v].y;
                        Su[v].x += q[v].x; Su[v].y += q[v].y;
                        Sv[v].x = fmaf(da, pa[v].x, fmaf(db, pb[v].x, Sv[v].x));
                        Sv[v].y = fmaf(da, pa[v].y, fmaf(db, pb[v].y, Sv[v].y));
                    }
                }
            } else
            for (int cy = r_lo; cy <= r_hi; ++cy) {
                float dy[kV], dyo2[kV];
                int c_lo = INT_MAX, c_hi = INT_MIN;
#pragma unroll
                for (int v = 0; v < kV; ++v) {
                    dy[v] = hy[v] - (float)(cy - wy[v]);
                    const float dyo = dy[v] * ov;
                    dyo2[v] = fmaf(dyo, dyo, 1e-20f);
                    const float rem = fmaf(-dy[v], dy[v], rmax2);
                    if (rem > 0.f) {
                        // r <= rho_max keeps the span inside the staged box
                        const float r = fminf(rem * rsqrt_fast(rem), rmax);
                        const int a_lo = max(0, (int)floorf(hx[v] - r) + 1);
                        const int a_hi = min(S - 1, (int)ceilf(hx[v] + r) - 1);
                        if (a_lo <= a_hi) {
                            c_lo = min(c_lo, wx[v] + a_lo);
                            c_hi = max(c_hi, wx[v] + a_hi);
                        }
                    }
                }
                if (c_lo > c_hi) continue;
                float dxo[kV], pr[kV], pi[kV], qr[kV], qi[kV];
#pragma unroll
                for (int v = 0; v < kV; ++v) {
                    dxo[v] = __fmul_rn(hx[v] - (float)(c_lo - wx[v]), ov);
                    pr[v] = pi[v] = qr[v] = qi[v] = 0.f;
                }
                row_taps<kV>(sh.tile + cy * kTile + c_lo, c_hi - c_lo + 1, dxo, dyo2, ov, tab_adj, pr, pi, qr, qi);
#pragma unroll
                for (int v = 0; v < kV; ++v) {
                    S0[v].x += pr[v]; S0[v].y += pi[v];
                    Su[v].x += qr[v]; Su[v].y += qi[v];
                    Sv[v].x = fmaf(dy[v], pr[v], Sv[v].x);
                    Sv[v].y = fmaf(dy[v], pi[v], Sv[v].y);
                }
            }
        } else {
            // unstaged: taps read the grid (L1/L2), the cell half of the ramp
            // comes from phx / phy; rows and columns are clipped to the grid
#pragma unroll
            for (int v = 0; v < kV; ++v) {
                const float2 *lo = kW ? a.grid + (size_t)wpl[v] * a.ng * a.ng : a.grid, *hi = lo + (size_t)a.ng * a.ng;    // kW: the two planes
                const int b_lo = max(max(0, (int)floorf(hy[v] - rmax) + 1), -iy0[v]);
                const int b_hi = min(min(S - 1, (int)ceilf(hy[v] + rmax) - 1), a.ng - 1 - iy0[v]);
                for (int b = b_lo; b <= b_hi; ++b) {
                    const float dy = hy[v] - (float)b;
                    const float rem = fmaf(-dy, dy, rmax2);
                    if (!(rem > 0.f)) continue;
                    const float r = fminf(rem * rsqrt_fast(rem), rmax);
                    const int a_lo = max(max(0, (int)floorf(hx[v] - r) + 1), -ix0[v]);
                    const int a_hi = min(min(S - 1, (int)ceilf(hx[v] + r) - 1), a.ng - 1 - ix0[v]);
                    const float dyo = dy * ov;
                    const float dyo2 = fmaf(dyo, dyo, 1e-20f);
                    float pr = 0.f, pi = 0.f, qr = 0.f, qi = 0.f;
                    const size_t row = (size_t)(iy0[v] + b) * a.ng + ix0[v];
                    float dd = __fmul_rn(hx[v] - (float)a_lo, ov);
                    for (int aa = a_lo; aa <= a_hi; ++aa, dd = __fsub_rn(dd, ov)) {
                        float2 gc;
                        if constexpr (kW) {
                            const float2 g0 = __ldg(&lo[row + aa]);
                            const float2 g1 = __ldg(&hi[row + aa]);
                            gc = make_float2(fmaf(wf[v], g1.x - g0.x, g0.x), fmaf(wf[v], g1.y - g0.y, g0.y));
                        } else {
                            gc = grid_cell(a, row + aa);
                        }
                        const float2 g = cmul(gc, sh.phx[aa]);
                        const float s2 = fmaf(dd, dd, dyo2);
                        const float tv = sqrt_fast(s2);
                        const float tf = __fadd_rz(tv, 8388608.0f);
                        const float2 e = lds_f2(tab_adj + ((unsigned)__float_as_int(tf) << 3));
                        const float A = fmaf(tv, e.y, e.x);
                        pr = fmaf(A, g.x, pr);
                        pi = fmaf(A, g.y, pi);
                        const float Ad = __fmul_rn(A, dd);
                        qr = fmaf(Ad, g.x, qr);
                        qi = fmaf(Ad, g.y, qi);
                    }
                    const float2 py = sh.phy[b];
                    const float2 P = cmul(make_float2(pr, pi), py);
                    const float2 Q = cmul(make_float2(qr, qi), py);
                    S0[v].x += P.x; S0[v].y += P.y;
                    Su[v].x += Q.x; Su[v].y += Q.y;
                    Sv[v].x = fmaf(dy, P.x, Sv[v].x);
                    Sv[v].y = fmaf(dy, P.y, Sv[v].y);
                }
            }
        }
        const float inv_ov = 1.0f / ov;
#pragma unroll
        for (int v = 0; v < kV; ++v) {                       // Q was accumulated with dx * ov
            Su[v].x *= inv_ov; Su[v].y *= inv_ov;
        }
    }

    // ---- epilogue: visibility half of the ramp, decorrelation, derivatives ----
    if (!active) return;
    const float al2 = a.chan[c].alpha2;
    float D = 1.f, el = 0.f, em = 0.f;
    if (a.decorrelation) {
        D = expf(-0.5f * al2 * (dL * dL + dM * dM));
        el = -dL * al2;                      // (l_j - l_i) alpha^2
        em = -dM * al2;
    }
    const float pi_f = 3.14159265358979f;
#pragma unroll
    for (int v = 0; v < kV; ++v) {
        const int t = t0 + v;
        if (t >= a.nt) break;
        const int ox = staged ? bx0 : ix0[v];
        const int oy = staged ? by0 : iy0[v];
        const float ph_arg = a.du * (((float)(ix0[v] - ox) + hx[v]) * L + ((float)(iy0[v] - oy) + hy[v]) * M);
        float s, co;
        sincospif(ph_arg, &s, &co);
        const float2 ph = make_float2(co, s);
        const float2 T0 = cmul(ph, S0[v]);
        float2 Tu = cmul(ph, Su[v]), Tv = cmul(ph, Sv[v]);
        Tu.x *= a.du; Tu.y *= a.du;          // tap offsets in wavelengths
        Tv.x *= a.du; Tv.y *= a.du;
        const float2 V = make_float2(D * T0.x, D * T0.y);
        // d/dl_i = D [(l_j - l_i) a^2 T0 + i pi Tu]; d/dl_j flips the first term; m likewise
        const float2 dli = make_float2(D * (el * T0.x - pi_f * Tu.y), D * (el * T0.y + pi_f * Tu.x));
        const float2 dmi = make_float2(D * (em * T0.x - pi_f * Tv.y), D * (em * T0.y + pi_f * Tv.x));
        const float2 dlj = make_float2(D * (-el * T0.x - pi_f * Tu.y), D * (-el * T0.y + pi_f * Tu.x));
        const float2 dmj = make_float2(D * (-em * T0.x - pi_f * Tv.y), D * (-em * T0.y + pi_f * Tv.x));
        const size_t k = ((size_t)t * a.n_bl + bl) * a.nc + c;
        if constexpr (kPredict) {
            a.vis_out[k] = V;
            if (a.dvis_out != nullptr) {
                const size_t plane = (size_t)a.nt * a.n_bl * a.nc;
                a.dvis_out[k] = dli;
                a.dvis_out[plane + k] = dmi;
                a.dvis_out[2 * plane + k] = dlj;
                a.dvis_out[3 * plane + k] = dmj;
            }
        } else {
            const float2 vo = a.vis_obs[k];
            const float w = a.w_scale * (a.w != nullptr ? a.w[k] : 1.f);
            const float2 R = make_float2(vo.x - V.x, vo.y - V.y);
            const float w2 = 2.f * w;
            acc[0] += w * (R.x * R.x + R.y * R.y);
            acc[1] -= w2 * (R.x * dli.x + R.y * dli.y);
            acc[2] -= w2 * (R.x * dmi.x + R.y * dmi.y);
            acc[3] -= w2 * (R.x * dlj.x + R.y * dlj.y);
            acc[4] -= w2 * (R.x * dmj.x + R.y * dmj.y);
            acc[5] += w2 * (dli.x * dli.x + dli.y * dli.y);
            acc[6] += w2 * (dli.x * dmi.x + dli.y * dmi.y);
            acc[7] += w2 * (dmi.x * dmi.x + dmi.y * dmi.y);
            acc[8] += w2 * (dlj.x * dlj.x + dlj.y * dlj.y);
            acc[9] += w2 * (dlj.x * dmj.x + dlj.y * dmj.y);
            acc[10] += w2 * (dmj.x * dmj.x + dmj.y * dmj.y);
            acc[11] += w2 * (dli.x * dlj.x + dli.y * dlj.y);
            acc[12] += w2 * (dli.x * dmj.x + dli.y * dmj.y);
            acc[13] += w2 * (dmi.x * dlj.x + dmi.y * dlj.y);
            acc[14] += w2 * (dmi.x * dmj.x + dmi.y * dmj.y);
        }
    }
}

// One launch covers either one context (queue == nullptr: block b handles
// brick b of a0) or a batch of contexts (persistent: each block pulls global
// brick numbers from an atomic queue until all sum(bricks) are taken; prefix
// holds the first global brick of each context).  Every brick writes its own
// partial record, so the result does not depend on which block ran it.
// The stacked instantiation (kW) asks for 3 blocks of kMaxThreads per SM, i.e. at
// most 85 registers; a minimum of 0 leaves the co-planar instantiations with the
// plain bound.
// kSplit: the instantiation that also runs split items (its co-planar contexts
// without them take the same code as before, at this kernel's registers).
template <bool kPredict, bool kW, bool kSplit>
__global__ void __launch_bounds__(kMaxThreads, kW || kSplit ? 3 : 0) eval_kernel(const EvalArgs a0, const EvalArgs *__restrict__ args,
                                                           const long long *__restrict__ prefix, int n_ctx,
                                                           unsigned long long *queue) {
    extern __shared__ __align__(16) float2 s_tab[];   // c_group * tab_stride, then split_taps' arrays (16-byte aligned)
    __shared__ BlockSharedT<!kW> sh;
    __shared__ EvalArgs s_a;
    __shared__ long long s_work, s_first;
    __shared__ int s_done;
    const bool persistent = queue != nullptr;
    long long next = -1;                              // thread 0: prefetched queue entry
    int cur = -1;                                     // thread 0: context whose arguments s_a holds
    for (;;) {
    if (persistent) {
        __syncthreads();                              // the previous brick is done with shared memory
        if (threadIdx.x == 0) {
            const long long gb = next >= 0 ? next : (long long)atomicAdd(queue, 1ull);
            next = (long long)atomicAdd(queue, 1ull);  // consumed next round: its latency overlaps this brick
            const long long end = prefix[n_ctx];
            s_done = gb >= end;
            if (gb < end) {
                // a block's bricks come in increasing order: the context is the
                // current one unless gb has passed its end
                if (cur < 0 || gb < prefix[cur] || gb >= prefix[cur + 1]) {
                    int lo = 0, hi = n_ctx - 1;       // last context with prefix[k] <= gb
                    while (lo < hi) {
                        const int mid = (lo + hi + 1) >> 1;
                        if (prefix[mid] <= gb) lo = mid; else hi = mid - 1;
                    }
                    cur = lo;
                    s_a = args[lo];                   // copied once per context change
                    s_first = prefix[lo];
                }
                s_work = gb;
            }
        }
        __syncthreads();
        if (s_done) return;
    } else {
        if (threadIdx.x == 0) s_a = a0;
        __syncthreads();
    }
    const EvalArgs &a = s_a;
    if (!(a.skip != nullptr && *a.skip)) {
    const int tid = threadIdx.x;
    const int qbrick = persistent ? (int)(s_work - s_first) : (int)blockIdx.x;
    // launch order -> brick (baseline groups permuted for locality when bl_order is set)
    const int brick = a.bl_order != nullptr ? a.bl_order[qbrick / a.bpb] * a.bpb + qbrick % a.bpb : qbrick;
    float acc[kRed];
#pragma unroll
    for (int k = 0; k < kRed; ++k) acc[k] = 0.f;
    float4 *s_split = reinterpret_cast<float4 *>(s_tab + (a.c_group * a.tab_stride + 1) / 2 * 2);
    // the stack's tile starts after the tables, whatever their number (a multiple of 16 bytes)
    float2 *s_wtile = s_tab + ((a.flat > 0 ? a.ch_span : a.c_group) * a.tab_stride + 1) / 2 * 2;
    bool active = false;                              // this thread holds a visibility
    if (kSplit && a.split > 1) eval_brick<kPredict, 1, kW, kSplit>(a, brick, s_tab, sh, s_split, nullptr, acc, active);
    else if (a.kv == 2) eval_brick<kPredict, 2, kW, false>(a, brick, s_tab, sh, nullptr, s_wtile, acc, active);
    else eval_brick<kPredict, 1, kW, false>(a, brick, s_tab, sh, nullptr, s_wtile, acc, active);
    if constexpr (!kPredict) {
        // ---- block reduction: a butterfly within each warp -- compensated
        // (Knuth's TwoSum, the rounding errors summed beside) for chi^2 and the
        // gradient, plain FP32 for the normal blocks -- then FP64 across warps ----
        float comp[5] = {0.f, 0.f, 0.f, 0.f, 0.f};
        // few warps of a split brick hold visibilities (the others' sums are zeros)
        const bool any = !kSplit || __any_sync(0xffffffffu, active);
#pragma unroll
        for (int o = any ? 16 : 0; o > 0; o >>= 1) {
#pragma unroll
            for (int k = 0; k < 5; ++k) {
                const float so = __shfl_xor_sync(0xffffffffu, acc[k], o);
                const float co = __shfl_xor_sync(0xffffffffu, comp[k], o);
                const float t = __fadd_rn(acc[k], so);
                const float bp = __fsub_rn(t, acc[k]);
                const float err = __fadd_rn(__fsub_rn(acc[k], __fsub_rn(t, bp)), __fsub_rn(so, bp));
                acc[k] = t;
                comp[k] = __fadd_rn(__fadd_rn(comp[k], co), err);
            }
#pragma unroll
            for (int k = 5; k < kRed; ++k) acc[k] += __shfl_xor_sync(0xffffffffu, acc[k], o);
        }
        const int warp = tid >> 5, lane = tid & 31;
        if (lane == 0) {
#pragma unroll
            for (int k = 0; k < kRed; ++k) sh.red[warp][k] = acc[k];
#pragma unroll
            for (int k = 0; k < 5; ++k) sh.red_c[warp][k] = comp[k];
        }
        __syncthreads();
        if (tid < kRed) {
            double s = 0.0;
            const int nw = (blockDim.x + 31) >> 5;
            for (int wi = 0; wi < nw; ++wi) {
                s += (double)sh.red[wi][tid];
                if (tid < 5) s += (double)sh.red_c[wi][tid];
            }
            a.partials[(size_t)tid * a.n_bricks + brick] = s;      // [kRed][n_bricks]
        }
    }
    }                                                 // not skipped
    if (!persistent) return;
    }                                                 // brick loop
}

// Second stage (a): per-baseline sums over its bricks, kL threads per
// (baseline, sum).  partials is [kRed][n_bricks] with the bricks of baseline bl
// at [bl * bpb, (bl + 1) * bpb).  The order of the additions is the same for
// either kL (eight strided sums, then a tree), so results do not depend on what
// else a batch holds.  Batched form: the global baseline number runs over the
// baselines of all contexts (bl_prefix).
// kL = 8 where a baseline has more than 8 records: its chain of dependent loads
// is what the pass costs (351 baselines of 300
// records: 52 us by one thread, 10 us by 8).
template <int kL>
__global__ void bl_reduce_kernel(const RedArgs r0, const RedArgs *__restrict__ ra,
                                 const int *__restrict__ bl_prefix, int n_ctx) {
    const long long gt = ((long long)blockIdx.x * blockDim.x + threadIdx.x) / kL;
    const int l = threadIdx.x % kL;
    const int gb = (int)(gt / kRed), k = (int)(gt - (long long)gb * kRed);
    RedArgs r = r0;
    int bl = gb;
    if (ra != nullptr) {
        if (gb >= bl_prefix[n_ctx]) return;
        int lo = 0, hi = n_ctx - 1;
        while (lo < hi) {
            const int mid = (lo + hi + 1) >> 1;
            if (bl_prefix[mid] <= gb) lo = mid; else hi = mid - 1;
        }
        r = ra[lo];
        bl = gb - bl_prefix[lo];
    }
    if (bl >= r.n_bl) return;
    if (r.skip != nullptr && *r.skip) return;
    const size_t nb = (size_t)r.n_bl * r.bpb;
    const double *p = r.partials + (size_t)k * nb + (size_t)bl * r.bpb;
    double sum;
    if constexpr (kL == 8) {
        sum = 0.0;
        for (int b = l; b < r.bpb; b += 8) sum += p[b];
        const unsigned group = 0xffu << (threadIdx.x & 24);
#pragma unroll
        for (int o = 4; o > 0; o >>= 1) sum += __shfl_xor_sync(group, sum, o);
    } else if (r.bpb == 1) {
        sum = p[0];
    } else {
        double s[8] = {0.0, 0.0, 0.0, 0.0, 0.0, 0.0, 0.0, 0.0};
        for (int b0 = 0; b0 < r.bpb; b0 += 8)
#pragma unroll
            for (int j = 0; j < 8; ++j)
                if (b0 + j < r.bpb) s[j] += p[b0 + j];
        sum = ((s[0] + s[4]) + (s[2] + s[6])) + ((s[1] + s[5]) + (s[3] + s[7]));
    }
    if (l == 0) r.blsum[(size_t)bl * kRed + k] = sum;
}

// Second stage (b): chi^2, per-antenna gradient and diagonal blocks, cross
// blocks; ev = chi2 | g[2n] | H[3n] | X[4 nbl].  blockIdx.x indexes ra when
// batched; blockIdx.y = 0 sums chi^2, the other blocks take a warp per antenna
// (its lanes over the partners, then a butterfly) and share the cross blocks.
// Fixed order.  One block per context, a thread per antenna, took 199 us at 197
// antennas and 17 us at 27: 15 and 6 now.
constexpr int kEvWarps = 8;
__global__ void __launch_bounds__(32 * kEvWarps) ev_kernel(const RedArgs r0, const RedArgs *__restrict__ ra) {
    const RedArgs r = ra != nullptr ? ra[blockIdx.x] : r0;
    if (r.skip != nullptr && *r.skip) return;
    const int tid = threadIdx.x, lane = tid & 31, warp = tid >> 5;
    const int n_ant = r.n_ant, n_bl = r.n_bl;
    if (blockIdx.y == 0) {
        __shared__ double s_chi[32 * kEvWarps];
        double chi = 0.0;
#pragma unroll 4
        for (int bl = tid; bl < n_bl; bl += 32 * kEvWarps) chi += r.blsum[(size_t)bl * kRed];
        s_chi[tid] = chi;
        __syncthreads();
        for (int o = 16 * kEvWarps; o > 0; o >>= 1) {
            if (tid < o) s_chi[tid] += s_chi[tid + o];
            __syncthreads();
        }
        if (tid == 0) r.ev[0] = s_chi[0];
        return;
    }
    // as many blocks as this context's antennas fill, whatever else the batch holds
    const int by = blockIdx.y - 1, nby = (n_ant + kEvWarps - 1) / kEvWarps;
    if (by >= nby) return;
    for (int bl = by * 32 * kEvWarps + tid; bl < n_bl; bl += nby * 32 * kEvWarps) {
        const double *sb = r.blsum + (size_t)bl * kRed;
        double *x = r.ev + 1 + 5 * (size_t)n_ant + 4 * (size_t)bl;
        x[0] = sb[11]; x[1] = sb[12]; x[2] = sb[13]; x[3] = sb[14];
    }
    const int an = by * kEvWarps + warp;
    if (an >= n_ant) return;
    double v[5] = {0.0, 0.0, 0.0, 0.0, 0.0};
    for (int o = lane; o < n_ant; o += 32) {
        if (o == an) continue;
        const int i = min(an, o), j = max(an, o);
        const int bl = i * (2 * n_ant - i - 1) / 2 + (j - i - 1);
        const double *sb = r.blsum + (size_t)bl * kRed + (an == i ? 0 : 2);
        v[0] += sb[1];
        v[1] += sb[2];
        sb += an == i ? 0 : 1;
        v[2] += sb[5];
        v[3] += sb[6];
        v[4] += sb[7];
    }
#pragma unroll
    for (int o = 16; o > 0; o >>= 1)
#pragma unroll
        for (int k = 0; k < 5; ++k) v[k] += __shfl_xor_sync(0xffffffffu, v[k], o);
    if (lane == 0) {
        r.ev[1 + 2 * an] = v[0];
        r.ev[2 + 2 * an] = v[1];
        double *h = r.ev + 1 + 2 * (size_t)n_ant + 3 * (size_t)an;
        h[0] = v[2]; h[1] = v[3]; h[2] = v[4];
    }
}

// Largest |uv(t+1) - uv(t)| over consecutive time steps and baselines (out_bits[0]) and
// largest |u| or |v| (out_bits[1]; infinity if any is not finite).
__global__ void step_max_kernel(const double *__restrict__ uvw, int nt, int n_bl, unsigned *out_bits) {
    float m = 0.f, far = 0.f;
    const long long n = (long long)nt * n_bl;
    for (long long k = blockIdx.x * (long long)blockDim.x + threadIdx.x; k < n; k += (long long)gridDim.x * blockDim.x) {
        const double *p = uvw + 3 * k;
        const float a = (float)fmax(fabs(p[0]), fabs(p[1]));
        far = isfinite(p[0] + p[1]) ? fmaxf(far, a) : INFINITY;
        if (k + n_bl >= n) continue;
        const double *q = p + 3 * (size_t)n_bl;
        const double du = q[0] - p[0], dv = q[1] - p[1];
        m = fmaxf(m, (float)sqrt(du * du + dv * dv));
    }
    for (int o = 16; o > 0; o >>= 1) {
        m = fmaxf(m, __shfl_xor_sync(0xffffffffu, m, o));
        far = fmaxf(far, __shfl_xor_sync(0xffffffffu, far, o));
    }
    if ((threadIdx.x & 31) == 0) {                    // both >= 0: bits order as values
        atomicMax(out_bits, __float_as_uint(m));
        atomicMax(out_bits + 1, __float_as_uint(far));
    }
}

__global__ void grid_to_bf16_kernel(const float2 *__restrict__ g, size_t n, unsigned *__restrict__ out) {
    for (size_t k = blockIdx.x * (size_t)blockDim.x + threadIdx.x; k < n; k += (size_t)gridDim.x * blockDim.x) {
        const __nv_bfloat162 b = __float22bfloat162_rn(g[k]);
        out[k] = *reinterpret_cast<const unsigned *>(&b);
    }
}

__global__ void split_uv_kernel(const double *__restrict__ uvw, size_t n, float4 *__restrict__ out) {
    for (size_t k = blockIdx.x * (size_t)blockDim.x + threadIdx.x; k < n; k += (size_t)gridDim.x * blockDim.x) {
        const double u = uvw[3 * k], v = uvw[3 * k + 1];
        const float uh = (float)u, vh = (float)v;
        out[k] = make_float4(uh, (float)(u - (double)uh), vh, (float)(v - (double)vh));
    }
}

}  // namespace

cudaError_t launch_split_uv(const double *uvw, size_t n, float4 *out, cudaStream_t s) {
    if (n == 0) return cudaSuccess;
    const int blocks = (int)std::min<size_t>((n + 255) / 256, 4096);
    split_uv_kernel<<<blocks, 256, 0, s>>>(uvw, n, out);
    return cudaGetLastError();
}

cudaError_t launch_grid_to_bf16(const float2 *grid, size_t n, unsigned *out, cudaStream_t s) {
    const int blocks = (int)std::min<size_t>((n + 255) / 256, 4096);
    grid_to_bf16_kernel<<<blocks, 256, 0, s>>>(grid, n, out);
    return cudaGetLastError();
}

cudaError_t launch_step_max(const double *uvw, int nt, int n_bl, unsigned *out_bits, cudaStream_t s) {
    const long long n = (long long)nt * n_bl;
    const int blocks = (int)std::min<long long>((n + 255) / 256, 1024);
    step_max_kernel<<<blocks, 256, 0, s>>>(uvw, nt, n_bl, out_bits);
    return cudaGetLastError();
}

size_t eval_dyn_smem(int c_group, int tab_stride) {
    return sizeof(float2) * (size_t)c_group * tab_stride;
}

// split_taps' share of a block's dynamic shared memory (and its alignment).
size_t eval_split_smem(int split, int support) {
    return split > 1 ? 16 + sizeof(float4) * (kMaxThreads + kMaxThreads * 6 / 4 + (size_t)(kMaxThreads / split) * support) : 0;
}

// The staged planes' share (and its alignment).
size_t eval_stack_smem(int wp_n) { return wp_n > 0 ? 16 + sizeof(float2) * kWCap : 0; }

cudaError_t launch_eval(const EvalArgs &a, bool predict, cudaStream_t s) {
    if (a.exact) return launch_exact(a, predict, s);
    const int threads = a.split > 1 ? kMaxThreads : ((a.flat > 0 ? a.flat : a.t_tile * a.c_group) + 31) / 32 * 32;
    const int blocks = (int)a.n_bricks;
    const size_t dyn = eval_dyn_smem(a.flat > 0 ? a.ch_span : a.c_group, a.tab_stride) + eval_split_smem(a.split, a.support) + eval_stack_smem(a.wp_n);
    if (a.wp_n > 0) {
        if (predict) eval_kernel<true, true, false><<<blocks, threads, dyn, s>>>(a, nullptr, nullptr, 0, nullptr);
        else eval_kernel<false, true, false><<<blocks, threads, dyn, s>>>(a, nullptr, nullptr, 0, nullptr);
    } else if (a.split > 1) {
        if (predict) eval_kernel<true, false, true><<<blocks, threads, dyn, s>>>(a, nullptr, nullptr, 0, nullptr);
        else eval_kernel<false, false, true><<<blocks, threads, dyn, s>>>(a, nullptr, nullptr, 0, nullptr);
    } else if (predict) {
        eval_kernel<true, false, false><<<blocks, threads, dyn, s>>>(a, nullptr, nullptr, 0, nullptr);
    } else {
        eval_kernel<false, false, false><<<blocks, threads, dyn, s>>>(a, nullptr, nullptr, 0, nullptr);
    }
    return cudaGetLastError();
}

cudaError_t launch_eval_batch(const EvalArgs *args_dev, const long long *prefix_dev, int n_ctx,
                              unsigned long long *queue, int threads, size_t dyn, int grid, bool stacked, bool split,
                              cudaStream_t s) {
    EvalArgs none{};
    if (stacked) eval_kernel<false, true, false><<<grid, threads, dyn, s>>>(none, args_dev, prefix_dev, n_ctx, queue);
    else if (split) eval_kernel<false, false, true><<<grid, threads, dyn, s>>>(none, args_dev, prefix_dev, n_ctx, queue);
    else eval_kernel<false, false, false><<<grid, threads, dyn, s>>>(none, args_dev, prefix_dev, n_ctx, queue);
    return cudaGetLastError();
}

cudaError_t eval_batch_occupancy(int threads, size_t dyn, bool stacked, bool split, int *blocks_per_sm) {
    if (stacked)
        return cudaOccupancyMaxActiveBlocksPerMultiprocessor(blocks_per_sm, eval_kernel<false, true, false>, threads, dyn);
    if (split)
        return cudaOccupancyMaxActiveBlocksPerMultiprocessor(blocks_per_sm, eval_kernel<false, false, true>, threads, dyn);
    return cudaOccupancyMaxActiveBlocksPerMultiprocessor(blocks_per_sm, eval_kernel<false, false, false>, threads, dyn);
}

// Dynamic shared memory the fused kernel can have on the current device: the
// opt-in limit less its static shared memory.
cudaError_t eval_smem_allowed(size_t *allowed) {
    int dev = 0, optin = 0;
    cudaError_t e = cudaGetDevice(&dev);
    if (e != cudaSuccess) return e;
    e = cudaDeviceGetAttribute(&optin, cudaDevAttrMaxSharedMemoryPerBlockOptin, dev);
    if (e != cudaSuccess) return e;
    cudaFuncAttributes fa{};
    e = cudaFuncGetAttributes(&fa, eval_kernel<false, false, false>);
    if (e != cudaSuccess) return e;
    *allowed = (size_t)optin > fa.sharedSizeBytes ? (size_t)optin - fa.sharedSizeBytes : 0;
    return cudaSuccess;
}

// Raises the fused kernel's dynamic shared-memory limit to everything the
// device allows beyond its static shared memory (never lowers it, so contexts
// with different channel groups can share the kernel), after checking that
// `dyn` bytes fit.
cudaError_t set_eval_smem(size_t dyn) {
    size_t allowed = 0;
    cudaError_t e = eval_smem_allowed(&allowed);
    if (e != cudaSuccess) return e;
    if (dyn > allowed) return cudaErrorInvalidValue;
    int dev = 0, optin = 0;
    e = cudaGetDevice(&dev);
    if (e == cudaSuccess) e = cudaDeviceGetAttribute(&optin, cudaDevAttrMaxSharedMemoryPerBlockOptin, dev);
    if (e != cudaSuccess) return e;
    for (const void *k : {(const void *)eval_kernel<true, false, false>, (const void *)eval_kernel<false, false, false>,
                          (const void *)eval_kernel<true, true, false>, (const void *)eval_kernel<false, true, false>,
                          (const void *)eval_kernel<true, false, true>, (const void *)eval_kernel<false, false, true>}) {
        // the stacked kernels hold a smaller static part, and more dynamic memory (eval_stack_smem)
        cudaFuncAttributes fa{};
        e = cudaFuncGetAttributes(&fa, k);
        if (e == cudaSuccess)
            e = cudaFuncSetAttribute(k, cudaFuncAttributeMaxDynamicSharedMemorySize, optin - (int)fa.sharedSizeBytes);
        if (e != cudaSuccess) return e;
    }
    return cudaSuccess;
}

namespace {
cudaError_t reduce_launches(const RedArgs &r, const RedArgs *ra_dev, const int *bl_prefix_dev, int n_ctx, int total_bl,
                            int max_bpb, int max_ant, cudaStream_t s) {
    const long long sums = (long long)total_bl * kRed;
    if (max_bpb > 8)
        bl_reduce_kernel<8><<<(unsigned)((8 * sums + 255) / 256), 256, 0, s>>>(r, ra_dev, bl_prefix_dev, n_ctx);
    else
        bl_reduce_kernel<1><<<(unsigned)((sums + 255) / 256), 256, 0, s>>>(r, ra_dev, bl_prefix_dev, n_ctx);
    cudaError_t e = cudaGetLastError();
    if (e != cudaSuccess) return e;
    ev_kernel<<<dim3(n_ctx, 1 + (max_ant + kEvWarps - 1) / kEvWarps), 32 * kEvWarps, 0, s>>>(r, ra_dev);
    return cudaGetLastError();
}
}  // namespace

cudaError_t launch_reduce(const RedArgs &r, cudaStream_t s) {
    return reduce_launches(r, nullptr, nullptr, 1, r.n_bl, r.bpb, r.n_ant, s);
}

cudaError_t launch_reduce_batch(const RedArgs *ra_dev, const int *bl_prefix_dev, int n_ctx, int total_bl, int max_bpb,
                                int max_ant, cudaStream_t s) {
    RedArgs none{};
    return reduce_launches(none, ra_dev, bl_prefix_dev, n_ctx, total_bl, max_bpb, max_ant, s);
}

}  // namespace psc
