// Model grid V° = F[I^M] of an image (Algorithm 1, first pre-compute; Eq. MEDD)
// by fast Fourier transforms, for the sizes that model_grid_fft_ok takes: the
// unnormalised DFT with sign exp(+2 pi i) of the N x N image zero-padded to
// Ng x Ng, as grid_dft.cu states it.
//
// Two passes, no workspace but the twiddle tables (of the powers of two: one
// constant table a context, filled once):
//   columns: the image is real, so columns c and c + 1 go through one complex
//     transform of length Ng (z = I_c + i I_{c+1}), of which the rows k = 0 ..
//     Ng/2 are kept (U[k][c]; the others are their conjugates);
//   rows: each kept row k is transformed once and written twice, as row k and,
//     reversed and conjugated, as row -k.
// U's row k is stored in the first N cells of the grid row that row k of the
// result takes.  The row pass reads only its own row before writing it and the
// row -k, which holds no part of U, so blocks need no order among themselves.
//
// One block per transform, the data in shared memory, Stockham passes of radix
// 16, 8, 4 or 2 (each thread holds 16 elements: one barrier before and one
// after the exchange, so a single buffer does), an odd part first as a direct
// DFT.  The exchange index is padded by one element in 16, which keeps the
// first passes' strided stores off one bank.  Twiddles come from FP64
// sincospi, rounded once, one contiguous table per pass.  The odd part's sums
// run in two levels of 16 terms.
//
// Bound: the grid's writes (8 Ng^2 bytes) and the shared-memory exchanges (three
// round trips of 8 Ng bytes per transform at Ng = 8192, two blocks an SM).
// 2048^2 -> 8192^2: columns 116 us, rows 228 us (2.4 TB/s of writes); one block
// an SM (95 registers a thread) took 90 us longer.  The call takes 359 us
// against 14,195 us for the DFT as matrix products on the tensor cores
// (grid_dft.cu, which grids of a long odd part still take), and its error
// against 64 bits is 0.9-1.6e-7 (relative L2, 128^2 to 8192^2 grids) against
// 1.5-4.1e-7.
#include <cuda.h>

#include <algorithm>
#include <cstdint>
#include <mutex>

#include "psc_internal.cuh"

namespace psc {
namespace {

constexpr int kE = 16;                // elements per thread
constexpr int kMaxPass = 5;           // ceil(log2(16384) / 3)
constexpr int kWide = 8192;           // longest transform that takes radix 16 (512 threads of up to 128 registers)

struct FftPlan {
    int n, odd, n_pass;
    int lr[kMaxPass], ns[kMaxPass], tw[kMaxPass];   // log2 radix, length done before the pass, table offset
    int tw_odd, tw_len;
};

FftPlan make_plan(int n) {
    const int n0 = n;
    FftPlan p{};
    p.n = n;
    int a = 0;
    while (n % 2 == 0) { n /= 2; ++a; }
    p.odd = n;
    const int most = n0 <= kWide ? 4 : 3;
    p.n_pass = (a + most - 1) / most;
    int ns = n, off = 0;
    for (int i = 0; i < p.n_pass; ++i) {
        const int left = p.n_pass - i;
        p.lr[i] = (a + left - 1) / left;               // as even a split as possible, the larger radices first
        a -= p.lr[i];
        p.ns[i] = ns;
        p.tw[i] = off;
        if (ns > 1) off += ((1 << p.lr[i]) - 1) * ns;
        ns <<= p.lr[i];
    }
    p.tw_odd = off;
    p.tw_len = off + (p.odd > 1 ? p.odd : 0);
    return p;
}

// Table entry (r - 1) ns + j of a pass: exp(2 pi i j r / (ns R)); of the odd part, entry k: exp(2 pi i k / odd).
__global__ void fft_twiddle_kernel(const FftPlan p, float2 *__restrict__ tw) {
    const int k = blockIdx.x * blockDim.x + threadIdx.x;
    if (k >= p.tw_len) return;
    double turns;
    if (k >= p.tw_odd) {
        turns = (double)(k - p.tw_odd) / p.odd;
    } else {
        int i = p.n_pass - 1;
        while (i > 0 && (k < p.tw[i] || p.ns[i] == 1)) --i;
        const int e = k - p.tw[i], r = e / p.ns[i] + 1, j = e % p.ns[i];
        turns = (double)((long long)j * r) / (double)((long long)p.ns[i] << p.lr[i]);
    }
    double s, c;
    sincospi(2.0 * turns, &s, &c);
    tw[k] = make_float2((float)c, (float)s);
}

__device__ __forceinline__ float2 cadd(float2 a, float2 b) { return make_float2(a.x + b.x, a.y + b.y); }
__device__ __forceinline__ float2 csub(float2 a, float2 b) { return make_float2(a.x - b.x, a.y - b.y); }
__device__ __forceinline__ float2 cmul(float2 a, float2 b) {
    return make_float2(fmaf(a.x, b.x, -a.y * b.y), fmaf(a.x, b.y, a.y * b.x));
}
__device__ __forceinline__ float2 mul_i(float2 a) { return make_float2(-a.y, a.x); }

// In-place transforms of R values, sign +, natural order in and out.
template <int R>
__device__ __forceinline__ void fft_r(float2 (&v)[R]);

template <>
__device__ __forceinline__ void fft_r<2>(float2 (&v)[2]) {
    const float2 a = v[0];
    v[0] = cadd(a, v[1]);
    v[1] = csub(a, v[1]);
}

template <>
__device__ __forceinline__ void fft_r<4>(float2 (&v)[4]) {
    const float2 s0 = cadd(v[0], v[2]), d0 = csub(v[0], v[2]);
    const float2 s1 = cadd(v[1], v[3]), d1 = mul_i(csub(v[1], v[3]));
    v[0] = cadd(s0, s1);
    v[1] = cadd(d0, d1);
    v[2] = csub(s0, s1);
    v[3] = csub(d0, d1);
}

template <>
__device__ __forceinline__ void fft_r<8>(float2 (&v)[8]) {
    float2 e[4] = {v[0], v[2], v[4], v[6]}, o[4] = {v[1], v[3], v[5], v[7]};
    fft_r<4>(e);
    fft_r<4>(o);
    const float h = 0.70710678118654752f;
    o[1] = make_float2(h * (o[1].x - o[1].y), h * (o[1].x + o[1].y));
    o[2] = mul_i(o[2]);
    o[3] = make_float2(-h * (o[3].x + o[3].y), h * (o[3].x - o[3].y));
#pragma unroll
    for (int k = 0; k < 4; ++k) {
        v[k] = cadd(e[k], o[k]);
        v[k + 4] = csub(e[k], o[k]);
    }
}

template <>
__device__ __forceinline__ void fft_r<16>(float2 (&v)[16]) {
    // 16 = 4 x 4: transforms over stride 4, twiddles exp(2 pi i a b / 16), transforms over stride 1
    const float c1 = 0.92387953251128674f, s1 = 0.38268343236508977f, h = 0.70710678118654752f;
    float2 t[4][4];
#pragma unroll
    for (int a = 0; a < 4; ++a) {
#pragma unroll
        for (int b = 0; b < 4; ++b) t[a][b] = v[a + 4 * b];
        fft_r<4>(t[a]);
    }
    t[1][1] = cmul(t[1][1], make_float2(c1, s1));
    t[1][2] = cmul(t[1][2], make_float2(h, h));
    t[1][3] = cmul(t[1][3], make_float2(s1, c1));
    t[2][1] = cmul(t[2][1], make_float2(h, h));
    t[2][2] = mul_i(t[2][2]);
    t[2][3] = cmul(t[2][3], make_float2(-h, h));
    t[3][1] = cmul(t[3][1], make_float2(s1, c1));
    t[3][2] = cmul(t[3][2], make_float2(-h, h));
    t[3][3] = cmul(t[3][3], make_float2(-c1, -s1));
#pragma unroll
    for (int b = 0; b < 4; ++b) {
        float2 u[4] = {t[0][b], t[1][b], t[2][b], t[3][b]};
        fft_r<4>(u);
#pragma unroll
        for (int a = 0; a < 4; ++a) v[b + 4 * a] = u[a];
    }
}

__device__ __forceinline__ int pad(int i) { return i + (i >> 4); }

// One Stockham pass of radix R: butterfly b takes elements b + r n / R, and
// leaves element r of its result at (b / ns) ns R + b % ns + r ns.  kPow2: ns
// is a power of two.
template <int R, bool kPow2, class Load, class Store>
__device__ __forceinline__ void fft_pass(int tid, int n, int ns, const float2 *__restrict__ tw, Load load, Store store) {
    constexpr int kB = kE / R;
    const int nb = n / R;
    float2 v[kB][R];
#pragma unroll
    for (int i = 0; i < kB; ++i) {
        // a thread past the last butterfly repeats it and stores nothing (a
        // branch here costs the registers twice and spills)
        const int b = min(tid + i * (int)blockDim.x, nb - 1);
#pragma unroll
        for (int r = 0; r < R; ++r) v[i][r] = load(b + r * nb);
        if (ns > 1) {
            const float2 *t = tw + (kPow2 ? b & (ns - 1) : b % ns);
#pragma unroll
            for (int r = 1; r < R; ++r) {
                v[i][r] = cmul(v[i][r], __ldg(t));
                t += ns;
            }
        }
        fft_r<R>(v[i]);
    }
    __syncthreads();
#pragma unroll
    for (int i = 0; i < kB; ++i) {
        const int b = tid + i * blockDim.x;
        if (b < nb) {
            const int j = kPow2 ? b & (ns - 1) : b % ns;
            int o = (b - j) * R + j;
#pragma unroll
            for (int r = 0; r < R; ++r) {
                store(o, v[i][r]);
                o += ns;
            }
        }
    }
    __syncthreads();
}

template <bool k16, bool kPow2, class Load, class Store>
__device__ __forceinline__ void fft_pass_any(int lr, int tid, int n, int ns, const float2 *tw, Load load, Store store) {
    switch (lr) {
        case 1: fft_pass<2, kPow2>(tid, n, ns, tw, load, store); break;
        case 2: fft_pass<4, kPow2>(tid, n, ns, tw, load, store); break;
        case 3: fft_pass<8, kPow2>(tid, n, ns, tw, load, store); break;
        default:
            if constexpr (k16) fft_pass<16, kPow2>(tid, n, ns, tw, load, store);
    }
}

// The transform of one block: elements from `load` (position 0 .. n - 1), results to `store` (frequency).
template <bool k16, bool kPow2, class Load, class Store>
__device__ __forceinline__ void fft_block(const FftPlan &p, const float2 *__restrict__ tw, float2 *buf, Load load,
                                          Store store) {
    auto rd = [&](int i) { return buf[pad(i)]; };
    auto wr = [&](int i, float2 v) { buf[pad(i)] = v; };
    if constexpr (!kPow2) {
        for (int i = threadIdx.x; i < p.n; i += blockDim.x) wr(i, load(i));
        __syncthreads();
        const int nb = p.n / p.odd;
        const float2 *w = tw + p.tw_odd;
        float2 v[kE];
#pragma unroll
        for (int i = 0; i < kE; ++i) {
            const int o = threadIdx.x + i * blockDim.x;
            float2 sum = make_float2(0.f, 0.f);
            if (o < p.n) {
                const int q = o / nb, j = o - q * nb;
                int k = 0;
                for (int s0 = 0; s0 < p.odd; s0 += 16) {
                    float2 part = make_float2(0.f, 0.f);
                    for (int s = s0; s < min(s0 + 16, p.odd); ++s) {
                        const float2 x = rd(j + s * nb), z = __ldg(&w[k]);
                        part.x = fmaf(x.x, z.x, fmaf(-x.y, z.y, part.x));
                        part.y = fmaf(x.x, z.y, fmaf(x.y, z.x, part.y));
                        k += q;
                        if (k >= p.odd) k -= p.odd;
                    }
                    sum = cadd(sum, part);
                }
            }
            v[i] = sum;
        }
        __syncthreads();
#pragma unroll
        for (int i = 0; i < kE; ++i) {
            const int o = threadIdx.x + i * blockDim.x;
            if (o < p.n) {
                const int q = o / nb, j = o - q * nb;
                wr(j * p.odd + q, v[i]);
            }
        }
        __syncthreads();
    }
    for (int i = 0; i < p.n_pass; ++i) {
        const bool first = kPow2 && i == 0, last = i == p.n_pass - 1;
        const float2 *t = tw + p.tw[i];
        // opaque to the compiler, which would otherwise hoist every radix's
        // addresses out of this loop and spill them
        int n = p.n, tid = threadIdx.x;
        asm volatile("" : "+r"(n), "+r"(tid));
        if (first && last) fft_pass_any<k16, kPow2>(p.lr[i], tid, n, p.ns[i], t, load, store);
        else if (first) fft_pass_any<k16, kPow2>(p.lr[i], tid, n, p.ns[i], t, load, wr);
        else if (last) fft_pass_any<k16, kPow2>(p.lr[i], tid, n, p.ns[i], t, rd, store);
        else fft_pass_any<k16, kPow2>(p.lr[i], tid, n, p.ns[i], t, rd, wr);
    }
}

// Grid row that holds frequency k = 0 .. Ng/2 (Ng/2 is -Ng/2, the first row).
__device__ __forceinline__ int row_of(int k, int ng) { return k < ng / 2 ? k + ng / 2 : 0; }

// k16: transforms up to kWide long; kPow2: no odd part.
template <bool k16, bool kPow2>
__global__ void __launch_bounds__(k16 ? 512 : 1024, k16 ? 2 : 1) fft_cols_kernel(const FftPlan p, const float2 *__restrict__ tw,
                                                        const float *__restrict__ img, int n, float2 *__restrict__ G) {
    extern __shared__ float2 buf[];
    const int ng = p.n, c = 2 * blockIdx.x, shift = ng - n / 2;
    auto load = [&](int i) {                          // position i = (r - N/2) mod Ng
        const int r = i < ng - n / 2 ? i + n / 2 : i - shift;
        return r < n ? make_float2(img[(size_t)r * n + c], img[(size_t)r * n + c + 1]) : make_float2(0.f, 0.f);
    };
    fft_block<k16, kPow2>(p, tw, buf, load, [&](int i, float2 v) { buf[pad(i)] = v; });
    for (int k = threadIdx.x; k <= ng / 2; k += blockDim.x) {
        const float2 a = buf[pad(k)], b = buf[pad(k ? ng - k : 0)];
        float2 *o = G + (size_t)row_of(k, ng) * ng + c;
        o[0] = make_float2(0.5f * (a.x + b.x), 0.5f * (a.y - b.y));
        o[1] = make_float2(0.5f * (a.y + b.y), 0.5f * (b.x - a.x));
    }
}

template <bool k16, bool kPow2>
__global__ void __launch_bounds__(k16 ? 512 : 1024, k16 ? 2 : 1) fft_rows_kernel(const FftPlan p, const float2 *__restrict__ tw, int n, float2 *G) {
    extern __shared__ float2 buf[];
    const int ng = p.n, k = blockIdx.x, half = ng / 2, shift = ng - n / 2;
    float2 *row = G + (size_t)row_of(k, ng) * ng;
    float2 *mirror = k > 0 && k < half ? G + (size_t)(half - k) * ng : nullptr;
    auto load = [&](int i) {
        const int c = i < ng - n / 2 ? i + n / 2 : i - shift;
        return c < n ? row[c] : make_float2(0.f, 0.f);
    };
    // every load precedes the pass's first barrier, every store follows it
    auto store = [&](int i, float2 v) {               // frequency i mod Ng
        row[i < half ? i + half : i - half] = v;
        if (mirror != nullptr) mirror[i <= half ? half - i : ng + half - i] = make_float2(v.x, -v.y);
    };
    fft_block<k16, kPow2>(p, tw, buf, load, store);
}

size_t buf_bytes(int n) { return (size_t)(n + n / 16 + 1) * sizeof(float2); }

}  // namespace

// A direct DFT of the odd part costs that many complex multiply-adds per grid cell, about
// 3.4e-13 s each (half of the cells are computed), the matrix products N of them at
// 0.6e-13 s (N % 8 == 0, tensor cores) or 2.4e-13 s (else), and launches and passes over
// memory besides.  So transforms where (us as products and as transforms):
//   the grid is a power of two (512 -> 8192: 1884 and 268);
//   N % 8 == 0 and the odd part is at most N / 8 (128 -> 7680, 15: 514 and 654; 1024 ->
//     8128, 127: 3998 and 3460; 512 -> 8128: 1882 and 3232; 64 -> 8176, 511: 366 and
//     11733), 32 more up to 1024^2 grids, where launches count (512 -> 600, 75: 143 and 82),
//     8 less beyond kWide, where a block fills an SM (64 -> 9216, 9: 451 and 1007);
//   else, at most N / 2 (514 -> 8160, 255: 8110 and 6192; 30 -> 7680, 15: 506 and 656), 16
//     less beyond kWide (30 -> 9216, 9: 703 and 1009), or N for images whose error on the
//     FP32 units would reach 1e-6.
bool model_grid_fft_ok(int n_img, int n_grid) {
    const int odd = make_plan(n_grid).odd;
    if (odd == 1) return true;
    const bool wide = n_grid > kWide;
    if (n_img % 8 == 0) return 8 * odd <= n_img + (n_grid <= 1024 ? 256 : wide ? -64 : 0);
    return 2 * odd <= n_img - (wide ? 32 : 0) || (n_img > 512 && odd <= n_img);
}

// Tables of the sizes with an odd part, built by every call; none for powers of two.
size_t model_grid_fft_ws_bytes(int n_grid) {
    const FftPlan p = make_plan(n_grid);
    return p.odd == 1 ? 0 : sizeof(float2) * (size_t)p.tw_len;
}

int context_slot() {
    using CtxGetId = CUresult (*)(CUcontext, unsigned long long *);
    static std::mutex mu;
    static CtxGetId get_id = nullptr;
    static unsigned long long ids[kCtxSlots];
    static int n = 0;
    std::lock_guard<std::mutex> lk(mu);
    if (!get_id) {
        void *p = nullptr;
        cudaDriverEntryPointQueryResult q{};
        if (cudaGetDriverEntryPointByVersion("cuCtxGetId", &p, 12000, cudaEnableDefault, &q) != cudaSuccess ||
            q != cudaDriverEntryPointSuccess || !p)
            return -1;
        get_id = reinterpret_cast<CtxGetId>(p);
    }
    unsigned long long id = 0;
    if (cudaFree(nullptr) != cudaSuccess || get_id(nullptr, &id) != CUDA_SUCCESS) return -1;    // cudaFree: a current context
    for (int i = 0; i < n; ++i)
        if (ids[i] == id) return i;
    if (n == kCtxSlots) return -1;
    ids[n] = id;
    return n++;
}

namespace {
// Twiddle tables of every power of two: size n's at [n, 2n).  Allocating and
// building the table on each call cost 140 us of the 490 us that 2048^2 ->
// 8192^2 took; constants for the context's life cost 256 KB.
constexpr int kMaxLog = 14;
__device__ float2 g_pow2_tw[2 << kMaxLog];

// The current context's tables, filled and complete on return.
cudaError_t pow2_tables(float2 **out) {
    static std::mutex mu;
    static float2 *addr[kCtxSlots] = {};
    const int slot = context_slot();
    std::lock_guard<std::mutex> lk(mu);
    if (slot < 0 || !addr[slot]) {
        void *q = nullptr;
        cudaError_t e = cudaGetSymbolAddress(&q, g_pow2_tw);
        cudaStream_t s = nullptr;
        if (e == cudaSuccess) e = cudaStreamCreateWithFlags(&s, cudaStreamNonBlocking);
        if (e != cudaSuccess) return e;
        for (int a = 1; a <= kMaxLog; ++a) {
            const FftPlan p = make_plan(1 << a);
            if (p.tw_len > 0) fft_twiddle_kernel<<<(p.tw_len + 127) / 128, 128, 0, s>>>(p, (float2 *)q + p.n);
        }
        e = cudaGetLastError();
        if (e == cudaSuccess) e = cudaStreamSynchronize(s);
        cudaStreamDestroy(s);
        if (e != cudaSuccess) return e;
        *out = (float2 *)q;
        if (slot >= 0) addr[slot] = *out;
        return cudaSuccess;
    }
    *out = addr[slot];
    return cudaSuccess;
}

template <bool k16, bool kPow2>
cudaError_t fft_launch(const FftPlan &p, int n_img, const float *image, float2 *tw, float2 *grid_out, cudaStream_t s) {
    const size_t smem = buf_bytes(p.n);
    const int threads = std::max(64, ((p.n + kE - 1) / kE + 31) / 32 * 32);
    for (const void *k : {(const void *)fft_cols_kernel<k16, kPow2>, (const void *)fft_rows_kernel<k16, kPow2>}) {
        const cudaError_t e = allow_smem(k, smem);
        if (e != cudaSuccess) return e;
    }
    if (!kPow2) fft_twiddle_kernel<<<(p.tw_len + 127) / 128, 128, 0, s>>>(p, tw);
    fft_cols_kernel<k16, kPow2><<<n_img / 2, threads, smem, s>>>(p, tw, image, n_img, grid_out);
    fft_rows_kernel<k16, kPow2><<<p.n / 2 + 1, threads, smem, s>>>(p, tw, n_img, grid_out);
    return cudaGetLastError();
}
}  // namespace

cudaError_t model_grid_fft(int n_img, int n_grid, const float *image, void *ws, float2 *grid_out, cudaStream_t s) {
    const FftPlan p = make_plan(n_grid);
    float2 *tw = (float2 *)ws;
    if (p.odd == 1) {
        const cudaError_t e = pow2_tables(&tw);
        if (e != cudaSuccess) return e;
        tw += n_grid;
        return n_grid <= kWide ? fft_launch<true, true>(p, n_img, image, tw, grid_out, s)
                               : fft_launch<false, true>(p, n_img, image, tw, grid_out, s);
    }
    return n_grid <= kWide ? fft_launch<true, false>(p, n_img, image, tw, grid_out, s)
                           : fft_launch<false, false>(p, n_img, image, tw, grid_out, s);
}

}  // namespace psc
