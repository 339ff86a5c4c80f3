// The learned initial estimate's MLP on the GPU: forward, backward and AdamW
// (an addition to the paper's method, which starts the minimiser from zero or
// from earlier solutions).
//
// Network 52 -> 256 -> 256 -> 256 -> 2, GELU (0.5 x (1 + erf(x / sqrt 2)))
// after the hidden layers, input standardised by fixed (mu, s).  Flat FP32
// parameter vector: W1 [52][256], b1, W2 [256][256], b2, W3 [256][256], b3,
// W4 [256][2], b4, mu [52], s [52]; y = x W + b.  Loss (1/B) sum (y - t)^2.
//
// Precision: FP32 master weights and AdamW state; every GEMM operand is
// bfloat16 (weights, standardised input, GELU outputs, output gradients),
// multiplied on the 5th-generation tensor cores (tcgen05.mma, FP32
// accumulator in tensor memory) -- the two-column last layer, whose operands are
// rounded alike, on the FP32 units; biases, GELU, its derivative and the
// optimiser are FP32.
//
// Shape.  The network is small (0.9 GFLOP for a minibatch of 1024): what counts
// is the number of dependent launches and the operand staging.  So one kernel
// (chain_kernel) takes a block of rows through every layer, forwards and, in
// training, back to the first layer's output gradient; the row block is the N
// side of each MMA and the layer's features the M side, so that 32 rows fill all
// 128 tensor-memory lanes and many SMs share a minibatch.  Weights come as ready
// operand images (pack_kernel, once per update) by bulk copies that run behind
// the previous layer's epilogue.  The activations and output gradients are left
// transposed ([feature][row]), as the weight-gradient products need them: these
// run as a second kernel, split over rows, and a third adds the splits, the bias
// gradients and the loss in fixed order.
// Measured: 102 us for the gradient of 1024 rows with its copy to the host (1179
// as eleven GEMM launches with element-wise staging), of which the three kernels
// 53; 25 us of kernels for the forward pass of 8192 rows (350).
#include <cuda_bf16.h>

#include <algorithm>
#include <cmath>
#include <cstdint>
#include <string>
#include <vector>

#include "psc_internal.cuh"

namespace psc {
namespace {

constexpr int kIn = 52, kHid = 256, kOut = 2;
constexpr size_t oW1 = 0, ob1 = oW1 + (size_t)kIn * kHid, oW2 = ob1 + kHid, ob2 = oW2 + (size_t)kHid * kHid,
                 oW3 = ob2 + kHid, ob3 = oW3 + (size_t)kHid * kHid, oW4 = ob3 + kHid, ob4 = oW4 + (size_t)kHid * kOut,
                 omu = ob4 + kOut, os = omu + kIn, kNParams = os + kIn, kNTrained = omu;

typedef __nv_bfloat16 bf16;

constexpr int kThreads = 256;
constexpr long kWaitLimit = 1L << 24;       // mbarrier polls before a kernel gives up (sets *err)
constexpr int kInP = 64;                    // the input layer's depth, padded with zeros
// Operand images of the weights: two halves of 128 features (M), each with its 8 x 8
// core matrices (8 features x 16 bytes of K) in K columns kColW bytes apart.
constexpr int kColW = 128 * 16;
constexpr size_t kImg1 = 2 * (size_t)(kInP / 8) * kColW, kImg = 2 * (size_t)(kHid / 8) * kColW;
constexpr size_t oF1 = 0, oF2 = oF1 + kImg1, oF3 = oF2 + kImg, oG3 = oF3 + kImg, oG2 = oG3 + kImg, kImages = oG2 + kImg;

__device__ __forceinline__ float gelu_f(float z) { return 0.5f * z * (1.0f + erff(z * 0.70710678118654752f)); }

__device__ __forceinline__ float gelu_grad_f(float z) {
    return 0.5f * (1.0f + erff(z * 0.70710678118654752f)) + z * expf(-0.5f * z * z) * 0.3989422804014327f;
}

// Shared-memory matrix descriptor of tcgen05.mma for a K-major operand in the
// no-swizzle core-matrix layout: core matrices of 8 rows x 16 bytes, those
// adjacent along K `lbo` bytes apart, those adjacent along M/N 128 bytes
// apart (descriptor version 1, layout type 0).
__device__ __forceinline__ uint64_t smem_desc(uint32_t saddr, uint32_t lbo) {
    return (uint64_t)((saddr >> 4) & 0x3FFF) | ((uint64_t)((lbo >> 4) & 0x3FFF) << 16) |
           ((uint64_t)(128 >> 4) << 32) | ((uint64_t)1 << 46);
}

// kind::f16 instruction descriptor: D FP32, A and B bfloat16, both K-major, M = 128, N = n.
__device__ __forceinline__ constexpr uint32_t mma_desc(int n) {
    return (1u << 4) | (1u << 7) | (1u << 10) | ((uint32_t)(n >> 3) << 17) | ((uint32_t)(128 >> 4) << 24);
}

__device__ __forceinline__ uint32_t saddr(const void *p) { return (uint32_t)__cvta_generic_to_shared(p); }

__device__ __forceinline__ void mbar_init(uint32_t mb) { asm volatile("mbarrier.init.shared::cta.b64 [%0], 1;" :: "r"(mb)); }

__device__ __forceinline__ bool mbar_wait(uint32_t addr, uint32_t parity) {
    for (long it = 0; it < kWaitLimit; ++it) {
        uint32_t ok;
        asm volatile("{\n.reg .pred q;\nmbarrier.try_wait.parity.shared::cta.b64 q, [%1], %2;\nselp.u32 %0, 1, 0, q;\n}"
                     : "=r"(ok) : "r"(addr), "r"(parity) : "memory");
        if (ok) return true;
    }
    return false;
}

// One contiguous bulk copy into shared memory, completing on mbarrier mb.
__device__ __forceinline__ void bulk_load(uint32_t dst, const void *src, uint32_t bytes, uint32_t mb) {
    asm volatile("mbarrier.arrive.expect_tx.shared::cta.b64 _, [%0], %1;" :: "r"(mb), "r"(bytes) : "memory");
    asm volatile("cp.async.bulk.shared::cluster.global.mbarrier::complete_tx::bytes [%0], [%1], %2, [%3];"
                 :: "r"(dst), "l"(reinterpret_cast<uint64_t>(src)), "r"(bytes), "r"(mb) : "memory");
}

__device__ __forceinline__ void tc_mma(uint32_t tmem, uint64_t ad, uint64_t bd, uint32_t idesc, uint32_t accum) {
    asm volatile("{\n.reg .pred p;\nsetp.ne.b32 p, %4, 0;\n"
                 "tcgen05.mma.cta_group::1.kind::f16 [%0], %1, %2, %3, p;\n}"
                 :: "r"(tmem), "l"(ad), "l"(bd), "r"(idesc), "r"(accum));
}

__device__ __forceinline__ void tc_commit(uint32_t mb) {
    asm volatile("tcgen05.commit.cta_group::1.mbarrier::arrive::one.shared::cluster.b64 [%0];" :: "r"(mb));
}

__device__ __forceinline__ void tc_ld16(uint32_t taddr, float *v) {
    uint32_t r[16];
    asm volatile("tcgen05.ld.sync.aligned.32x32b.x16.b32 {%0,%1,%2,%3,%4,%5,%6,%7,%8,%9,%10,%11,%12,%13,%14,%15}, [%16];"
                 : "=r"(r[0]), "=r"(r[1]), "=r"(r[2]), "=r"(r[3]), "=r"(r[4]), "=r"(r[5]), "=r"(r[6]), "=r"(r[7]),
                   "=r"(r[8]), "=r"(r[9]), "=r"(r[10]), "=r"(r[11]), "=r"(r[12]), "=r"(r[13]), "=r"(r[14]), "=r"(r[15])
                 : "r"(taddr));
    asm volatile("tcgen05.wait::ld.sync.aligned;");
#pragma unroll
    for (int j = 0; j < 16; ++j) v[j] = __uint_as_float(r[j]);
}

__device__ __forceinline__ uint32_t pack2(float lo, float hi) {
    const __nv_bfloat162 b = __floats2bfloat162_rn(lo, hi);
    return *reinterpret_cast<const uint32_t *>(&b);
}

// The operand images of the current weights: F = (feature out, feature in) for
// the forward layers, G = (feature in, feature out) for the way back.
__global__ void pack_kernel(const float *__restrict__ p, unsigned char *__restrict__ img) {
    const int chunk = blockIdx.x * blockDim.x + threadIdx.x;      // one 16-byte row of a core matrix
    if (chunk >= (int)(kImages / 16)) return;
    const size_t byte = (size_t)chunk * 16;
    const bool first = byte < oF2;
    const int which = first ? 0 : 1 + (int)((byte - oF2) / kImg);  // F1, F2, F3, G3, G2
    const size_t in = first ? byte : (byte - oF2) % kImg;
    const int depth = first ? kInP : kHid;
    const size_t half_bytes = (size_t)(depth / 8) * kColW;
    const int half = (int)(in / half_bytes);
    const int rest = (int)(in % half_bytes);
    const int k0 = rest / kColW * 8, m = half * 128 + rest % kColW / 16;
    const float *w = p + (which == 0 ? oW1 : which == 1 || which == 4 ? oW2 : oW3);
    float v[8];
#pragma unroll
    for (int j = 0; j < 8; ++j) {
        const int k = k0 + j;
        if (which >= 3) v[j] = w[(size_t)m * kHid + k];
        else v[j] = which > 0 || k < kIn ? w[(size_t)k * kHid + m] : 0.f;
    }
    *reinterpret_cast<uint4 *>(img + byte) = make_uint4(pack2(v[0], v[1]), pack2(v[2], v[3]), pack2(v[4], v[5]), pack2(v[6], v[7]));
}

struct ChainArgs {
    const float *p;            // parameters (biases, last layer, standardisation)
    const unsigned char *img;  // operand images
    const float *x, *t;        // [B][52], [B][2] (training)
    int B;
    float *y;                  // [B][2]
    int *err;
    // training outputs, rows of ld elements (ld a multiple of 64, at least the rows of all blocks)
    size_t ld;
    bf16 *aT;                  // [64 | 256 | 256][ld] standardised input, GELU outputs of layers 1 and 2
    bf16 *dT;                  // [3][256][ld] output gradients of layers 1, 2, 3
    float *zT;                 // [2][256][ld] layers 1 and 2 before the GELU
    float *part;               // [blocks][kPart] bias gradients of layers 1..3, the last layer's gradients
    double *lossp;             // [blocks]
};
constexpr int kPart = 3 * kHid + kHid * kOut + kOut;

// kN rows of the batch per block.
template <int kN>
constexpr size_t chain_smem() {
    return kImg1 + kImg + (size_t)(kHid / 8) * (kN * 16 + 16) + 128;
}

// The rows of one block through the network.  Thread (half, f): feature 128 half
// + f of every layer, all kN rows.  Tensor memory: columns [half kN, ..).
template <int kN, bool kTrain>
__global__ void __launch_bounds__(kThreads, 1) chain_kernel(const ChainArgs a) {
    extern __shared__ unsigned char raw[];
    __shared__ __align__(8) uint64_t s_bar[3];
    __shared__ uint32_t s_tmem;
    __shared__ float s_y[kN][kOut];          // outputs, then (training) their gradients
    constexpr uint32_t kColB = kN * 16 + 16;                 // K columns of the activations: 16 bytes of padding spread the banks
    constexpr uint32_t kCols = 2 * kN < 32 ? 32 : 2 * kN;
    const int tid = threadIdx.x, warp = tid >> 5, lane = tid & 31;
    const int half = warp >> 2, f = tid;                     // f = 128 half + 32 (warp & 3) + lane
    const int b0 = blockIdx.x * kN;
    const uint32_t base = (saddr(raw) + 127u) & ~127u;
    const uint32_t sW1 = base, sW = sW1 + (uint32_t)kImg1, sAct = sW + (uint32_t)kImg;
    unsigned char *act = raw + (sAct - saddr(raw));
    const uint32_t wb1 = saddr(&s_bar[0]), wb = saddr(&s_bar[1]), mb = saddr(&s_bar[2]);
    if (tid == 0) {
        mbar_init(wb1);
        mbar_init(wb);
        mbar_init(mb);
        asm volatile("fence.mbarrier_init.release.cluster;");
        bulk_load(sW1, a.img + oF1, (uint32_t)kImg1, wb1);
        bulk_load(sW, a.img + oF2, (uint32_t)kImg, wb);
    }
    if (warp == 0) {
        asm volatile("tcgen05.alloc.cta_group::1.sync.aligned.shared::cta.b32 [%0], %1;" :: "r"(saddr(&s_tmem)), "r"(kCols));
        asm volatile("tcgen05.relinquish_alloc_permit.cta_group::1.sync.aligned;");
    }
    // standardised input as the first layer's N operand (rows past the batch: zero)
    for (int e = tid; e < kN * kInP; e += kThreads) {
        const int n = e / kInP, k = e % kInP;
        float v = 0.f;
        if (k < kIn && b0 + n < a.B) v = (a.x[(size_t)(b0 + n) * kIn + k] - a.p[omu + k]) / a.p[os + k];
        *reinterpret_cast<bf16 *>(act + (k >> 3) * kColB + n * 16 + (k & 7) * 2) = __float2bfloat16(v);
    }
    asm volatile("fence.proxy.async.shared::cta;");
    asm volatile("tcgen05.fence::before_thread_sync;");
    __syncthreads();
    asm volatile("tcgen05.fence::after_thread_sync;");
    const uint32_t tmem = s_tmem;
    const uint32_t my_tmem = tmem + ((uint32_t)(32 * (warp & 3)) << 16) + (uint32_t)(half * kN);
    if constexpr (kTrain) {
        // the same, transposed, for the first layer's weight gradient
        for (int e = tid; e < kInP * kN / 8; e += kThreads) {
            const int k = e / (kN / 8), n0 = e % (kN / 8) * 8;
            alignas(16) bf16 v[8];
#pragma unroll
            for (int j = 0; j < 8; ++j) v[j] = *reinterpret_cast<const bf16 *>(act + (k >> 3) * kColB + (n0 + j) * 16 + (k & 7) * 2);
            *reinterpret_cast<uint4 *>(a.aT + (size_t)k * a.ld + b0 + n0) = *reinterpret_cast<const uint4 *>(v);
        }
    }
    uint32_t wpar = 0;                       // parity of the next weight copy into sW
    uint32_t mpar = 0;                       // parity of the next MMA commit
    bool ok = true, pending = true;          // pending: a copy into sW not yet waited for
    // one layer's product: D[half] = image[half] (128 x depth) x act (depth x kN); then the
    // next image's copy, and the wait for the MMAs
    auto product = [&](uint32_t img, int depth, uint32_t wbar, uint32_t par, const unsigned char *next) {
        if (tid == 0) {
            ok = mbar_wait(wbar, par);
            if (ok) {
                asm volatile("tcgen05.fence::after_thread_sync;");
                for (int h = 0; h < 2; ++h)
                    for (int k = 0; k < depth; k += 16)
                        tc_mma(tmem + (uint32_t)(h * kN), smem_desc(img + (uint32_t)((h * depth + k) / 8 * kColW), kColW),
                               smem_desc(sAct + (uint32_t)(k / 8) * kColB, kColB), mma_desc(kN), k > 0);
                tc_commit(mb);
            }
        }
        ok = __syncthreads_and(ok);          // thread 0's wait decides for all
        if (!ok) return;
        ok = mbar_wait(mb, mpar);
        mpar ^= 1u;
        ok = __syncthreads_and(ok);
        if (!ok) return;
        asm volatile("tcgen05.fence::after_thread_sync;");
        if (next != nullptr) {               // the image is free: its MMAs are done
            if (tid == 0) bulk_load(sW, next, (uint32_t)kImg, wb);
            pending = true;
        }
    };
    float v[kN];
    uint32_t packed[kN / 2];                 // bfloat16 pairs of consecutive rows
    auto load_acc = [&]() {
#pragma unroll
        for (int c = 0; c < kN; c += 16) tc_ld16(my_tmem + (uint32_t)c, v + c);
    };
    // the packed values as the next product's N operand, and transposed to global memory
    auto put = [&](bf16 *out) {
#pragma unroll
        for (int n = 0; n < kN; n += 2) {
            unsigned char *q = act + (f >> 3) * kColB + n * 16 + (f & 7) * 2;
            *reinterpret_cast<unsigned short *>(q) = (unsigned short)(packed[n / 2] & 0xFFFFu);
            *reinterpret_cast<unsigned short *>(q + 16) = (unsigned short)(packed[n / 2] >> 16);
        }
        if (out != nullptr) {
            uint4 *o = reinterpret_cast<uint4 *>(out + (size_t)f * a.ld + b0);
#pragma unroll
            for (int n = 0; n < kN; n += 8) o[n / 8] = make_uint4(packed[n / 2], packed[n / 2 + 1], packed[n / 2 + 2], packed[n / 2 + 3]);
        }
    };
    auto publish = [&]() {                   // shared-memory stores before the next product's MMAs
        asm volatile("fence.proxy.async.shared::cta;");
        asm volatile("tcgen05.fence::before_thread_sync;");
        __syncthreads();
        asm volatile("tcgen05.fence::after_thread_sync;");
    };
    // ---- forwards ----
    for (int L = 1; L <= 3; ++L) {
        if (L == 1) {
            product(sW1, kInP, wb1, 0, nullptr);
        } else {
            product(sW, kHid, wb, wpar, L == 2 ? a.img + oF3 : kTrain ? a.img + oG3 : nullptr);
            if (L == 3 && !kTrain) pending = false;
            wpar ^= 1u;
        }
        if (!ok) break;
        load_acc();
        const float bias = a.p[(L == 1 ? ob1 : L == 2 ? ob2 : ob3) + f];
#pragma unroll
        for (int n = 0; n < kN; ++n) v[n] += bias;
        if (kTrain && L < 3) {
            float4 *z = reinterpret_cast<float4 *>(a.zT + ((size_t)(L - 1) * kHid + f) * a.ld + b0);
#pragma unroll
            for (int n = 0; n < kN; n += 4) z[n / 4] = make_float4(v[n], v[n + 1], v[n + 2], v[n + 3]);
        }
#pragma unroll
        for (int n = 0; n < kN; n += 2) packed[n / 2] = pack2(gelu_f(v[n]), gelu_f(v[n + 1]));
        put(kTrain && L < 3 ? a.aT + (size_t)(kInP + (L - 1) * kHid) * a.ld : nullptr);
        publish();
    }
    // ---- last layer: y = a3 W4 + b4, a warp per row, lanes over features ----
    if (ok) {
        float w4[8][kOut];
#pragma unroll
        for (int j = 0; j < 8; ++j)
#pragma unroll
            for (int o = 0; o < kOut; ++o) w4[j][o] = __bfloat162float(__float2bfloat16(a.p[oW4 + (size_t)(8 * lane + j) * kOut + o]));
        double l = 0.0;
        for (int n = warp; n < kN; n += kThreads / 32) {
            const uint4 q = *reinterpret_cast<const uint4 *>(act + lane * kColB + n * 16);
            const uint32_t u[4] = {q.x, q.y, q.z, q.w};
            float s[kOut] = {0.f, 0.f};
#pragma unroll
            for (int j = 0; j < 8; ++j) {
                const float x = __uint_as_float(j & 1 ? u[j / 2] & 0xFFFF0000u : u[j / 2] << 16);
#pragma unroll
                for (int o = 0; o < kOut; ++o) s[o] = fmaf(x, w4[j][o], s[o]);
            }
#pragma unroll
            for (int o = 16; o > 0; o >>= 1)
#pragma unroll
                for (int k = 0; k < kOut; ++k) s[k] += __shfl_xor_sync(0xffffffffu, s[k], o);
            if (lane < kOut) {
                float y = (lane == 0 ? s[0] : s[1]) + a.p[ob4 + lane];
                const bool in = b0 + n < a.B;
                const size_t e = (size_t)(b0 + n) * kOut + lane;
                if (in && a.y != nullptr) a.y[e] = y;
                if constexpr (kTrain) {
                    const float d = in ? y - a.t[e] : 0.f;
                    l += (double)d * d;
                    s_y[n][lane] = 2.0f * d / (float)a.B;
                }
            }
        }
        if constexpr (kTrain) {
            l += __shfl_down_sync(0xffffffffu, l, 1);
            __shared__ double s_loss[kThreads / 32];
            if (lane == 0) s_loss[warp] = l;
            __syncthreads();
            if (tid == 0) {
                double tot = 0.0;
                for (int w = 0; w < kThreads / 32; ++w) tot += s_loss[w];
                a.lossp[blockIdx.x] = tot;
            }
            // ---- backwards.  Layer 3: dz = (dy W4^T) gelu'(z), z still in v ----
            float *part = a.part + (size_t)blockIdx.x * kPart;
            const float w0 = __bfloat162float(__float2bfloat16(a.p[oW4 + (size_t)f * kOut]));
            const float w1 = __bfloat162float(__float2bfloat16(a.p[oW4 + (size_t)f * kOut + 1]));
            float db = 0.f, g0 = 0.f, g1 = 0.f, d0s = 0.f, d1s = 0.f;
#pragma unroll
            for (int n = 0; n < kN; n += 2) {
                float dz[2];
#pragma unroll
                for (int j = 0; j < 2; ++j) {
                    const float d0 = s_y[n + j][0], d1 = s_y[n + j][1];
                    const float r0 = __bfloat162float(__float2bfloat16(d0)), r1 = __bfloat162float(__float2bfloat16(d1));
                    const float act3 = __uint_as_float(j ? packed[n / 2] & 0xFFFF0000u : packed[n / 2] << 16);
                    g0 = fmaf(act3, r0, g0);
                    g1 = fmaf(act3, r1, g1);
                    d0s += d0;
                    d1s += d1;
                    dz[j] = fmaf(r0, w0, r1 * w1) * gelu_grad_f(v[n + j]);
                    db += dz[j];
                }
                packed[n / 2] = pack2(dz[0], dz[1]);
            }
            part[2 * kHid + f] = db;
            part[3 * kHid + f * kOut] = g0;
            part[3 * kHid + f * kOut + 1] = g1;
            if (f < kOut) part[3 * kHid + kHid * kOut + f] = f ? d1s : d0s;
            put(a.dT + (size_t)2 * kHid * a.ld);
            publish();
            for (int L = 2; L >= 1 && ok; --L) {
                product(sW, kHid, wb, wpar, L == 2 ? a.img + oG2 : nullptr);
                if (L == 1) pending = false;
                wpar ^= 1u;
                if (!ok) break;
                load_acc();
                const float4 *z = reinterpret_cast<const float4 *>(a.zT + ((size_t)(L - 1) * kHid + f) * a.ld + b0);
                db = 0.f;
#pragma unroll
                for (int n = 0; n < kN; n += 4) {
                    const float4 zz = z[n / 4];
                    v[n] *= gelu_grad_f(zz.x);
                    v[n + 1] *= gelu_grad_f(zz.y);
                    v[n + 2] *= gelu_grad_f(zz.z);
                    v[n + 3] *= gelu_grad_f(zz.w);
                    db += (v[n] + v[n + 1]) + (v[n + 2] + v[n + 3]);
                    packed[n / 2] = pack2(v[n], v[n + 1]);
                    packed[n / 2 + 1] = pack2(v[n + 2], v[n + 3]);
                }
                part[(L - 1) * kHid + f] = db;
                put(a.dT + (size_t)(L - 1) * kHid * a.ld);
                publish();
            }
        }
    }
    if (!ok) {
        // a wait ran out: report it; copies and MMAs may still be in flight, so
        // wait once more (bounded) before the memory and TMEM are given up
        if (tid == 0) {
            atomicExch(a.err, 1);
            mbar_wait(wb1, 0);
            if (pending) mbar_wait(wb, wpar);
            mbar_wait(mb, mpar);
        }
        __syncthreads();
    }
    asm volatile("tcgen05.fence::before_thread_sync;");
    __syncthreads();
    if (warp == 0) asm volatile("tcgen05.dealloc.cta_group::1.sync.aligned.b32 %0, %1;" :: "r"(tmem), "r"(kCols));
}

// Weight gradients dW = X^T dZ of layers 1..3 as tiles of 128 inputs x 64 outputs
// over kKc rows at a time: blockIdx.x = tile (4 of layer 1, 8 each of layers 2 and
// 3), blockIdx.y = split of the rows.  Both operands are K-major as they lie.
constexpr int kKc = 256, kTiles = 20, kGN = 64;
constexpr size_t kSplitLd = (kNParams + 3) / 4 * 4;      // one split's sums, 16-byte aligned rows
constexpr uint32_t kColA2 = 128 * 16 + 16, kColB2 = kGN * 16 + 16;
constexpr size_t kWgSmem = (size_t)(kKc / 8) * (kColA2 + kColB2) + 128;

__global__ void __launch_bounds__(kThreads, 1) wgrad_kernel(const bf16 *__restrict__ aT, const bf16 *__restrict__ dT, size_t ld,
                                                            int rows, int per_split, float *__restrict__ out, int *err) {
    extern __shared__ unsigned char raw[];
    __shared__ __align__(8) uint64_t s_bar;
    __shared__ uint32_t s_tmem;
    const int tid = threadIdx.x, warp = tid >> 5, lane = tid & 31;
    const int tile = blockIdx.x;
    const int layer = tile < 4 ? 0 : tile < 12 ? 1 : 2;
    const int q = tile < 4 ? tile : (tile - 4) % 8;
    const int m0 = layer == 0 ? 0 : (q >> 2) * 128, n0 = (q & 3) * kGN;
    const int m_rows = layer == 0 ? kInP : 128;
    const bf16 *A = aT + (size_t)(layer == 0 ? 0 : kInP + (layer - 1) * kHid + m0) * ld;
    const bf16 *Bm = dT + (size_t)(layer * kHid + n0) * ld;
    const uint32_t sA = (saddr(raw) + 127u) & ~127u, sB = sA + (kKc / 8) * kColA2;
    unsigned char *pA = raw + (sA - saddr(raw)), *pB = raw + (sB - saddr(raw));
    const uint32_t mb = saddr(&s_bar);
    if (tid == 0) {
        mbar_init(mb);
        asm volatile("fence.mbarrier_init.release.cluster;");
    }
    if (warp == 0) {
        asm volatile("tcgen05.alloc.cta_group::1.sync.aligned.shared::cta.b32 [%0], %1;" :: "r"(saddr(&s_tmem)), "r"(kGN));
        asm volatile("tcgen05.relinquish_alloc_permit.cta_group::1.sync.aligned;");
    }
    asm volatile("tcgen05.fence::before_thread_sync;");
    __syncthreads();
    asm volatile("tcgen05.fence::after_thread_sync;");
    const uint32_t tmem = s_tmem;
    const int k_lo = blockIdx.y * per_split, k_hi = min(rows, k_lo + per_split);
    bool ok = true;
    uint32_t par = 0;
    const uint4 zero = make_uint4(0, 0, 0, 0);
    for (int k0 = k_lo; k0 < k_hi && ok; k0 += kKc) {
        // 16 bytes = 8 rows of the batch; rows past the batch's blocks read as zero
#pragma unroll 8
        for (int e = tid; e < 128 * (kKc / 8); e += kThreads) {
            const int m = e / (kKc / 8), c = e % (kKc / 8);
            *reinterpret_cast<uint4 *>(pA + c * kColA2 + m * 16) =
                m < m_rows && k0 + 8 * c < k_hi ? *reinterpret_cast<const uint4 *>(A + (size_t)m * ld + k0 + 8 * c) : zero;
        }
#pragma unroll 8
        for (int e = tid; e < kGN * (kKc / 8); e += kThreads) {
            const int n = e / (kKc / 8), c = e % (kKc / 8);
            *reinterpret_cast<uint4 *>(pB + c * kColB2 + n * 16) =
                k0 + 8 * c < k_hi ? *reinterpret_cast<const uint4 *>(Bm + (size_t)n * ld + k0 + 8 * c) : zero;
        }
        asm volatile("fence.proxy.async.shared::cta;");
        asm volatile("tcgen05.fence::before_thread_sync;");
        __syncthreads();
        asm volatile("tcgen05.fence::after_thread_sync;");
        if (tid == 0) {
            for (int k = 0; k < kKc; k += 16)
                tc_mma(tmem, smem_desc(sA + (uint32_t)(k / 8) * kColA2, kColA2), smem_desc(sB + (uint32_t)(k / 8) * kColB2, kColB2),
                       mma_desc(kGN), k0 > k_lo || k > 0);
            tc_commit(mb);
        }
        ok = mbar_wait(mb, par);
        par ^= 1u;
        ok = __syncthreads_and(ok);
    }
    if (!ok && tid == 0) {
        atomicExch(err, 1);
        mbar_wait(mb, par ^ 1u);
    }
    asm volatile("tcgen05.fence::after_thread_sync;");
    if (ok && k_lo < k_hi) {
        // warp w: accumulator rows 32 (w & 3) .., columns 32 (w >> 2) ..
        const int m = 32 * (warp & 3) + lane, c0 = 32 * (warp >> 2);
        float v[32];
        tc_ld16(tmem + ((uint32_t)(32 * (warp & 3)) << 16) + (uint32_t)c0, v);
        tc_ld16(tmem + ((uint32_t)(32 * (warp & 3)) << 16) + (uint32_t)(c0 + 16), v + 16);
        if (m < (layer == 0 ? kIn : 128)) {
            float4 *o = reinterpret_cast<float4 *>(out + (size_t)blockIdx.y * kSplitLd + (layer == 0 ? oW1 : layer == 1 ? oW2 : oW3) +
                                                   (size_t)(m0 + m) * kHid + n0 + c0);
#pragma unroll
            for (int j = 0; j < 32; j += 4) o[j / 4] = make_float4(v[j], v[j + 1], v[j + 2], v[j + 3]);
        }
    }
    asm volatile("tcgen05.fence::before_thread_sync;");
    __syncthreads();
    if (warp == 0) asm volatile("tcgen05.dealloc.cta_group::1.sync.aligned.b32 %0, %1;" :: "r"(tmem), "r"(kGN));
}

// The gradient: weights from their splits, biases and the last layer from the
// blocks' partial sums, in fixed order; and the loss.
__global__ void grad_sum_kernel(const float *__restrict__ splits, int n_split, const float *__restrict__ part,
                                const double *__restrict__ lossp, int blocks, int B, float *__restrict__ g, double *loss) {
    const size_t e = blockIdx.x * (size_t)blockDim.x + threadIdx.x;
    if (e == 0) {
        double l = 0.0;
        for (int b = 0; b < blocks; ++b) l += lossp[b];
        *loss = l / B;
    }
    if (e >= kNParams) return;
    float s = 0.f;
    int at = -1;                                       // place in a block's partial sums
    if (e >= ob1 && e < oW2) at = (int)(e - ob1);
    else if (e >= ob2 && e < oW3) at = kHid + (int)(e - ob2);
    else if (e >= ob3 && e < oW4) at = 2 * kHid + (int)(e - ob3);
    else if (e >= oW4 && e < omu) at = 3 * kHid + (int)(e - oW4);
    if (at >= 0) {
#pragma unroll 8
        for (int b = 0; b < blocks; ++b) s += part[(size_t)b * kPart + at];
    } else if (e < omu) {
#pragma unroll 4
        for (int k = 0; k < n_split; ++k) s += splits[(size_t)k * kSplitLd + e];
    }
    g[e] = s;
}

// AdamW (decoupled weight decay) on the trained parameters; c1, c2 are the
// bias corrections 1 - beta^step.
__global__ void adamw_kernel(float *p, const float *g, float *m, float *v, int n, float lr, float b1, float b2,
                             float eps, float wd, float c1, float c2) {
    for (int e = blockIdx.x * blockDim.x + threadIdx.x; e < n; e += gridDim.x * blockDim.x) {
        const float ge = g[e];
        const float me = b1 * m[e] + (1.f - b1) * ge;
        const float ve = b2 * v[e] + (1.f - b2) * ge * ge;
        m[e] = me;
        v[e] = ve;
        const float mh = me / c1, vh = ve / c2;
        const float pe = p[e] - lr * (mh / (sqrtf(vh) + eps) + wd * p[e]);
        p[e] = pe;
    }
}

int blocks_for(size_t n, int threads = 256) {
    size_t b = (n + threads - 1) / threads;
    return (int)(b > 4096 ? 4096 : (b < 1 ? 1 : b));
}

}  // namespace
}  // namespace psc

using namespace psc;

struct psc_mlp {
    cudaStream_t stream = nullptr;
    int max_batch = 0;
    float *p = nullptr, *g = nullptr, *m = nullptr, *v = nullptr;   // [kNParams]
    unsigned char *img = nullptr;    // operand images of the weights
    float *y = nullptr;              // [B][2]
    size_t ld = 0;                   // row length of the transposed buffers
    bf16 *aT = nullptr, *dT = nullptr;
    float *zT = nullptr, *part = nullptr, *splits = nullptr;
    double *lossp = nullptr;
    double *d_loss = nullptr;
    int *d_err = nullptr;            // set by a kernel whose tensor-core or copy wait ran out
    long long step = 0;
    std::vector<float> host;
    std::string err;
};

namespace {

psc_status mfail(psc_mlp *m, psc_status st, const std::string &msg) {
    if (m) m->err = msg;
    return set_global_error(st, msg.c_str());
}

#define PSC_MCUDA(mm, call)                                                                      \
    do {                                                                                         \
        cudaError_t e_ = (call);                                                                 \
        if (e_ != cudaSuccess)                                                                   \
            return mfail((mm), e_ == cudaErrorMemoryAllocation ? PSC_ERR_OOM : PSC_ERR_CUDA,     \
                         std::string(#call) + ": " + cudaGetErrorString(e_));                    \
    } while (0)

template <class T>
cudaError_t mall(T **p, size_t n) { return cudaMalloc((void **)p, sizeof(T) * (n ? n : 1)); }

// After a synchronisation: PSC_ERR_TIMEOUT (and the flag cleared) if a GEMM
// gave up waiting for its tensor-core work since the last check.
psc_status check_device_err(psc_mlp *m) {
    int h = 0;
    cudaError_t e = cudaMemcpy(&h, m->d_err, sizeof(int), cudaMemcpyDeviceToHost);
    if (e != cudaSuccess) return mfail(m, PSC_ERR_CUDA, std::string("device error flag: ") + cudaGetErrorString(e));
    if (h == 0) return PSC_OK;
    cudaMemset(m->d_err, 0, sizeof(int));
    return mfail(m, PSC_ERR_TIMEOUT, "a network kernel timed out waiting for its MMAs");
}

void mfree(psc_mlp *m) {
    if (!m) return;
    void *ptrs[] = {m->p, m->g, m->m, m->v, m->img, m->y, m->aT, m->dT, m->zT, m->part, m->splits, m->lossp,
                    m->d_loss, m->d_err};
    for (void *q : ptrs) cudaFree(q);
    delete m;
}

cudaError_t refresh_images(psc_mlp *m) {
    pack_kernel<<<(int)((kImages / 16 + 255) / 256), 256, 0, m->stream>>>(m->p, m->img);
    return cudaGetLastError();
}

// Rows of a block: 32 fill more SMs, 64 read the weights half as often.  The line
// lies where 32 rows would take a second wave of blocks (one per SM): 8192 rows
// forwards took 26.7 us as 256 blocks of 32 and 22.6 us as 128 of 64.
constexpr int kWideRows = 152 * 32;
int block_rows(int B) { return B > kWideRows ? 64 : 32; }
int n_blocks(int B) { return (B + block_rows(B) - 1) / block_rows(B); }
constexpr int kMaxSplit = 8;

template <int kN, bool kTrain>
cudaError_t launch_chain(const ChainArgs &a, cudaStream_t s) {
    const size_t smem = chain_smem<kN>();
    const cudaError_t e = cudaFuncSetAttribute(chain_kernel<kN, kTrain>, cudaFuncAttributeMaxDynamicSharedMemorySize, (int)smem);
    if (e != cudaSuccess) return e;
    chain_kernel<kN, kTrain><<<(a.B + kN - 1) / kN, kThreads, smem, s>>>(a);
    return cudaGetLastError();
}

ChainArgs chain_args(psc_mlp *m, const float *x, const float *t, int B, float *y) {
    ChainArgs a{};
    a.p = m->p; a.img = m->img;
    a.x = x; a.t = t; a.B = B; a.y = y;
    a.err = m->d_err;
    a.ld = m->ld; a.aT = m->aT; a.dT = m->dT; a.zT = m->zT;
    a.part = m->part; a.lossp = m->lossp;
    return a;
}

psc_status forward(psc_mlp *m, const float *x, int B, float *y) {
    const ChainArgs a = chain_args(m, x, nullptr, B, y);
    PSC_MCUDA(m, block_rows(B) == 64 ? (launch_chain<64, false>(a, m->stream)) : (launch_chain<32, false>(a, m->stream)));
    return PSC_OK;
}

// Loss and gradient of the batch (into m->g and m->d_loss).
psc_status gradient(psc_mlp *m, const float *x, const float *t, int B) {
    cudaStream_t s = m->stream;
    const ChainArgs a = chain_args(m, x, t, B, nullptr);
    PSC_MCUDA(m, block_rows(B) == 64 ? (launch_chain<64, true>(a, s)) : (launch_chain<32, true>(a, s)));
    const int blocks = n_blocks(B), rows = blocks * block_rows(B), chunks = (rows + kKc - 1) / kKc;
    const int per = (chunks + kMaxSplit - 1) / kMaxSplit * kKc, splits = (rows + per - 1) / per;
    PSC_MCUDA(m, cudaFuncSetAttribute(wgrad_kernel, cudaFuncAttributeMaxDynamicSharedMemorySize, (int)kWgSmem));
    wgrad_kernel<<<dim3(kTiles, splits), kThreads, kWgSmem, s>>>(m->aT, m->dT, m->ld, rows, per, m->splits, m->d_err);
    PSC_MCUDA(m, cudaGetLastError());
    grad_sum_kernel<<<(int)((kNParams + 255) / 256), 256, 0, s>>>(m->splits, splits, m->part, m->lossp, blocks, B, m->g, m->d_loss);
    PSC_MCUDA(m, cudaGetLastError());
    return PSC_OK;
}

psc_status check_batch(psc_mlp *m, const void *x, int B) {
    if (!m) return set_global_error(PSC_ERR_ARG, "mlp is NULL");
    if (!x) return mfail(m, PSC_ERR_ARG, "input is NULL");
    if (B < 1 || B > m->max_batch) return mfail(m, PSC_ERR_ARG, "batch must be in [1, max_batch]");
    return PSC_OK;
}

}  // namespace

extern "C" {

int psc_mlp_n_params(void) { return (int)kNParams; }

psc_status psc_mlp_create(psc_mlp **out, int max_batch, void *stream) {
    if (!out) return set_global_error(PSC_ERR_ARG, "out is NULL");
    *out = nullptr;
    if (max_batch < 1 || max_batch > (1 << 24)) return set_global_error(PSC_ERR_ARG, "max_batch must be in [1, 2^24]");
    psc_mlp *m = new psc_mlp();
    m->stream = (cudaStream_t)stream;
    m->max_batch = max_batch;
    const size_t B = max_batch;
    cudaError_t e = cudaSuccess;
    if (e == cudaSuccess) e = mall(&m->p, kNParams);
    if (e == cudaSuccess) e = mall(&m->g, kNParams);
    if (e == cudaSuccess) e = mall(&m->m, kNParams);
    if (e == cudaSuccess) e = mall(&m->v, kNParams);
    m->ld = (B + 63) / 64 * 64;
    if (e == cudaSuccess) e = mall(&m->img, kImages);
    if (e == cudaSuccess) e = mall(&m->y, B * kOut);
    if (e == cudaSuccess) e = mall(&m->aT, (size_t)(kInP + 2 * kHid) * m->ld);
    if (e == cudaSuccess) e = mall(&m->dT, (size_t)3 * kHid * m->ld);
    if (e == cudaSuccess) e = mall(&m->zT, (size_t)2 * kHid * m->ld);
    // blocks of 32 rows up to kWideRows, of 64 beyond
    const size_t blocks = std::max((std::min(B, (size_t)kWideRows) + 31) / 32, (B + 63) / 64);
    if (e == cudaSuccess) e = mall(&m->part, blocks * kPart);
    if (e == cudaSuccess) e = mall(&m->lossp, blocks);
    if (e == cudaSuccess) e = mall(&m->splits, (size_t)kMaxSplit * kSplitLd);
    if (e == cudaSuccess) e = mall(&m->d_loss, 1);
    if (e == cudaSuccess) e = mall(&m->d_err, 1);
    if (e == cudaSuccess) e = cudaMemsetAsync(m->d_err, 0, sizeof(int), m->stream);
    if (e != cudaSuccess) {
        mfree(m);
        return set_global_error(e == cudaErrorMemoryAllocation ? PSC_ERR_OOM : PSC_ERR_CUDA, "psc_mlp_create: allocation");
    }
    *out = m;
    return PSC_OK;
}

void psc_mlp_destroy(psc_mlp *m) { mfree(m); }

psc_status psc_mlp_set_params(psc_mlp *m, const float *params) {
    if (!m || !params) return set_global_error(PSC_ERR_ARG, "mlp and params must be non-NULL");
    for (int i = 0; i < kIn; ++i)
        if (!(params[os + i] > 0.f)) return mfail(m, PSC_ERR_ARG, "input scales s must be > 0");
    PSC_MCUDA(m, cudaMemcpyAsync(m->p, params, sizeof(float) * kNParams, cudaMemcpyHostToDevice, m->stream));
    PSC_MCUDA(m, cudaMemsetAsync(m->m, 0, sizeof(float) * kNParams, m->stream));
    PSC_MCUDA(m, cudaMemsetAsync(m->v, 0, sizeof(float) * kNParams, m->stream));
    PSC_MCUDA(m, refresh_images(m));
    PSC_MCUDA(m, cudaStreamSynchronize(m->stream));
    m->step = 0;
    return PSC_OK;
}

psc_status psc_mlp_get_params(psc_mlp *m, float *params) {
    if (!m || !params) return set_global_error(PSC_ERR_ARG, "mlp and params must be non-NULL");
    PSC_MCUDA(m, cudaMemcpyAsync(params, m->p, sizeof(float) * kNParams, cudaMemcpyDeviceToHost, m->stream));
    PSC_MCUDA(m, cudaStreamSynchronize(m->stream));
    return check_device_err(m);
}

psc_status psc_mlp_forward(psc_mlp *m, const float *x_dev, int batch, float *y_dev) {
    psc_status st = check_batch(m, x_dev, batch);
    if (st != PSC_OK) return st;
    if (!y_dev) return mfail(m, PSC_ERR_ARG, "output is NULL");
    const size_t y_bytes = sizeof(float) * (size_t)batch * kOut;
    const uintptr_t x0 = (uintptr_t)x_dev, y0 = (uintptr_t)y_dev;
    if (y0 >= x0 + sizeof(float) * (size_t)batch * kIn || x0 >= y0 + y_bytes) return forward(m, x_dev, batch, y_dev);
    // outputs inside the input's buffer: written once every block has read its rows
    st = forward(m, x_dev, batch, m->y);
    if (st != PSC_OK) return st;
    PSC_MCUDA(m, cudaMemcpyAsync(y_dev, m->y, y_bytes, cudaMemcpyDeviceToDevice, m->stream));
    return PSC_OK;
}

psc_status psc_mlp_grad(psc_mlp *m, const float *x_dev, const float *t_dev, int batch, float *grad_host, double *loss) {
    psc_status st = check_batch(m, x_dev, batch);
    if (st != PSC_OK) return st;
    if (!t_dev) return mfail(m, PSC_ERR_ARG, "targets are NULL");
    st = gradient(m, x_dev, t_dev, batch);
    if (st != PSC_OK) return st;
    if (grad_host) PSC_MCUDA(m, cudaMemcpyAsync(grad_host, m->g, sizeof(float) * kNParams, cudaMemcpyDeviceToHost, m->stream));
    if (loss) PSC_MCUDA(m, cudaMemcpyAsync(loss, m->d_loss, sizeof(double), cudaMemcpyDeviceToHost, m->stream));
    if (grad_host || loss) {
        PSC_MCUDA(m, cudaStreamSynchronize(m->stream));
        return check_device_err(m);
    }
    return PSC_OK;
}

psc_status psc_mlp_train_step(psc_mlp *m, const float *x_dev, const float *t_dev, int batch, double lr, double *loss) {
    psc_status st = check_batch(m, x_dev, batch);
    if (st != PSC_OK) return st;
    if (!t_dev) return mfail(m, PSC_ERR_ARG, "targets are NULL");
    if (!(lr > 0.0) || !std::isfinite(lr)) return mfail(m, PSC_ERR_ARG, "lr must be > 0");
    st = gradient(m, x_dev, t_dev, batch);
    if (st != PSC_OK) return st;
    m->step += 1;
    const float b1 = 0.9f, b2 = 0.999f;
    const float c1 = (float)(1.0 - std::pow(0.9, (double)m->step));
    const float c2 = (float)(1.0 - std::pow(0.999, (double)m->step));
    adamw_kernel<<<blocks_for(kNTrained), 256, 0, m->stream>>>(m->p, m->g, m->m, m->v, (int)kNTrained, (float)lr, b1, b2,
                                                               1e-8f, 1e-4f, c1, c2);
    PSC_MCUDA(m, cudaGetLastError());
    PSC_MCUDA(m, refresh_images(m));
    if (loss) {
        PSC_MCUDA(m, cudaMemcpyAsync(loss, m->d_loss, sizeof(double), cudaMemcpyDeviceToHost, m->stream));
        PSC_MCUDA(m, cudaStreamSynchronize(m->stream));
        return check_device_err(m);
    }
    return PSC_OK;
}

psc_status psc_mlp_infer_offsets(psc_mlp *m, const float *feat_dev, int n_ant, double sigma_prior_rad, double *lm_out) {
    psc_status st = check_batch(m, feat_dev, n_ant);
    if (st != PSC_OK) return st;
    if (!lm_out) return mfail(m, PSC_ERR_ARG, "lm_out is NULL");
    st = forward(m, feat_dev, n_ant, m->y);
    if (st != PSC_OK) return st;
    if (m->host.size() < (size_t)n_ant * kOut) m->host.resize((size_t)n_ant * kOut);
    PSC_MCUDA(m, cudaMemcpyAsync(m->host.data(), m->y, sizeof(float) * n_ant * kOut, cudaMemcpyDeviceToHost, m->stream));
    PSC_MCUDA(m, cudaStreamSynchronize(m->stream));
    st = check_device_err(m);
    if (st != PSC_OK) return st;
    for (int i = 0; i < n_ant * kOut; ++i) lm_out[i] = (double)m->host[i] * sigma_prior_rad;
    return PSC_OK;
}

}  // extern "C"
