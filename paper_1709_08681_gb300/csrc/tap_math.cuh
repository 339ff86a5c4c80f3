// Device helpers of the fused evaluation kernels (eval.cu, track.cu): complex
// products, hardware square roots, packed FP32x2 arithmetic, the grid
// position of a visibility from the FP32 split of its baseline, and the
// per-row tap loops of the kernel of Eq. AIJPOINTING (radial A° table in
// shared memory as intercept/slope pairs, the phase ramp factored out of the
// taps).  Internal; included by the .cu files only.
#pragma once

#include <cuda_runtime.h>

namespace psc {
namespace tap {

__device__ __forceinline__ float2 cmul(float2 a, float2 b) {
    return make_float2(a.x * b.x - a.y * b.y, a.x * b.y + a.y * b.x);
}

__device__ __forceinline__ float rsqrt_fast(float x) {
    float r;
    asm("rsqrt.approx.ftz.f32 %0, %1;" : "=f"(r) : "f"(x));
    return r;
}

__device__ __forceinline__ float sqrt_fast(float x) {
    float r;
    asm("sqrt.approx.ftz.f32 %0, %1;" : "=f"(r) : "f"(x));
    return r;
}

// (px, py) += a (gx, gy) as one packed FP32x2 FMA: each lane rounds exactly
// like fmaf, and the pair costs one instruction instead of two.
__device__ __forceinline__ void fma2_acc(float &px, float &py, float a, float gx, float gy) {
    asm("{\n.reg .b64 aa, gg, pp;\nmov.b64 aa, {%2, %2};\nmov.b64 gg, {%3, %4};\nmov.b64 pp, {%0, %1};\n"
        "fma.rn.f32x2 pp, aa, gg, pp;\nmov.b64 {%0, %1}, pp;\n}"
        : "+f"(px), "+f"(py) : "f"(a), "f"(gx), "f"(gy));
}

// Shared-memory load at a 32-bit shared address.  Not volatile: the loads
// are pure, and the compiler may schedule them early (they are only issued
// inside tap loops that follow the barrier publishing the tables).
__device__ __forceinline__ float2 lds_f2(unsigned addr) {
    float2 v;
    asm("ld.shared.v2.f32 {%0, %1}, [%2];" : "=f"(v.x), "=f"(v.y) : "r"(addr));
    return v;
}

// Grid position x = u sc + Ng/2 of a baseline coordinate given as two floats
// (u = uh + ul, metres) and the channel's scale sc = sh + sl, without FP64:
// the product's rounding error comes from an FMA (exact), the small cross
// terms are added to it, and Ng/2 is added with Knuth's TwoSum, whose error
// term is exact.  Returns floor(x) in n and x - floor(x) in f (rounded once
// to FP32).
__device__ __forceinline__ void grid_pos(float uh, float ul, float sh, float sl, float half, int &n, float &f) {
    // _rn intrinsics: no FMA contraction may merge these steps
    const float p = __fmul_rn(uh, sh);
    float e = fmaf(uh, sh, -p);
    e = fmaf(uh, sl, e);
    e = fmaf(ul, sh, e);
    const float s = __fadd_rn(half, p);
    const float bb = __fsub_rn(s, half);
    const float r = __fadd_rn(__fsub_rn(half, __fsub_rn(s, bb)), __fsub_rn(p, bb));
    const float fl = floorf(s);
    f = __fadd_rn(__fsub_rn(s, fl), __fadd_rn(r, e));     // s - fl is exact
    n = (int)fl;
    if (f < 0.f) { f += 1.f; n -= 1; }
    else if (f >= 1.f) { f -= 1.f; n += 1; }
}

// Packed FP32x2 helpers on float2 pairs (each lane rounds like the scalar op).
__device__ __forceinline__ float2 ffma2(float2 a, float2 b, float2 c) {
    float2 d;
    asm("{\n.reg .b64 aa, bb, cc;\nmov.b64 aa, {%2, %3};\nmov.b64 bb, {%4, %5};\nmov.b64 cc, {%6, %7};\n"
        "fma.rn.f32x2 cc, aa, bb, cc;\nmov.b64 {%0, %1}, cc;\n}"
        : "=f"(d.x), "=f"(d.y) : "f"(a.x), "f"(a.y), "f"(b.x), "f"(b.y), "f"(c.x), "f"(c.y));
    return d;
}
__device__ __forceinline__ float2 fmul2(float2 a, float2 b) {
    float2 d;
    asm("{\n.reg .b64 aa, bb;\nmov.b64 aa, {%2, %3};\nmov.b64 bb, {%4, %5};\n"
        "mul.rn.f32x2 aa, aa, bb;\nmov.b64 {%0, %1}, aa;\n}"
        : "=f"(d.x), "=f"(d.y) : "f"(a.x), "f"(a.y), "f"(b.x), "f"(b.y));
    return d;
}
__device__ __forceinline__ float2 fadd2(float2 a, float2 b) {
    float2 d;
    asm("{\n.reg .b64 aa, bb;\nmov.b64 aa, {%2, %3};\nmov.b64 bb, {%4, %5};\n"
        "add.rn.f32x2 aa, aa, bb;\nmov.b64 {%0, %1}, aa;\n}"
        : "=f"(d.x), "=f"(d.y) : "f"(a.x), "f"(a.y), "f"(b.x), "f"(b.y));
    return d;
}
__device__ __forceinline__ float2 fadd2_rz(float2 a, float2 b) {
    float2 d;
    asm("{\n.reg .b64 aa, bb;\nmov.b64 aa, {%2, %3};\nmov.b64 bb, {%4, %5};\n"
        "add.rz.f32x2 aa, aa, bb;\nmov.b64 {%0, %1}, aa;\n}"
        : "=f"(d.x), "=f"(d.y) : "f"(a.x), "f"(a.y), "f"(b.x), "f"(b.y));
    return d;
}

// Two neighbouring rows of taps for two visibilities, n cells from row_a and row_b,
// the visibilities' scalars packed in pairs (s2, floor(t) + 2^23, A dxo and the dxo step
// are one packed instruction for both): the same column offsets for both rows, twice
// the independent work per step of the sqrt -> table -> FMA chain that one row at a
// time waited for.  Returns each row's P = sum A G' (pa, pb) and both rows'
// Q = sum A dxo G'.
__device__ __forceinline__ void row_pair_taps2(const float2 *__restrict__ row_a, const float2 *__restrict__ row_b, int n,
                                               float2 dxo, float2 dyo2a, float2 dyo2b, float ov, unsigned tab_adj,
                                               float2 (&pa)[2], float2 (&pb)[2], float2 (&q)[2]) {
    const float2 step = make_float2(-ov, -ov);
    const float2 magic = make_float2(8388608.0f, 8388608.0f);
    pa[0] = pa[1] = pb[0] = pb[1] = q[0] = q[1] = make_float2(0.f, 0.f);
#pragma unroll 2
    for (int k = 0; k < n; ++k) {
        const float2 ga = row_a[k], gb = row_b[k];
        const float2 sa = ffma2(dxo, dxo, dyo2a), sb = ffma2(dxo, dxo, dyo2b);
        const float2 ta = make_float2(sqrt_fast(sa.x), sqrt_fast(sa.y));
        const float2 tb = make_float2(sqrt_fast(sb.x), sqrt_fast(sb.y));
        const float2 fa = fadd2_rz(ta, magic), fb = fadd2_rz(tb, magic);
        const float2 ea0 = lds_f2(tab_adj + ((unsigned)__float_as_int(fa.x) << 3));
        const float2 ea1 = lds_f2(tab_adj + ((unsigned)__float_as_int(fa.y) << 3));
        const float2 eb0 = lds_f2(tab_adj + ((unsigned)__float_as_int(fb.x) << 3));
        const float2 eb1 = lds_f2(tab_adj + ((unsigned)__float_as_int(fb.y) << 3));
        const float2 Aa = make_float2(fmaf(ta.x, ea0.y, ea0.x), fmaf(ta.y, ea1.y, ea1.x));
        const float2 Ab = make_float2(fmaf(tb.x, eb0.y, eb0.x), fmaf(tb.y, eb1.y, eb1.x));
        const float2 Ada = fmul2(Aa, dxo), Adb = fmul2(Ab, dxo);
        fma2_acc(pa[0].x, pa[0].y, Aa.x, ga.x, ga.y);
        fma2_acc(pa[1].x, pa[1].y, Aa.y, ga.x, ga.y);
        fma2_acc(pb[0].x, pb[0].y, Ab.x, gb.x, gb.y);
        fma2_acc(pb[1].x, pb[1].y, Ab.y, gb.x, gb.y);
        fma2_acc(q[0].x, q[0].y, Ada.x, ga.x, ga.y);
        fma2_acc(q[1].x, q[1].y, Ada.y, ga.x, ga.y);
        fma2_acc(q[0].x, q[0].y, Adb.x, gb.x, gb.y);
        fma2_acc(q[1].x, q[1].y, Adb.y, gb.x, gb.y);
        dxo = fadd2(dxo, step);
    }
}

// One row of taps for kV visibilities: n consecutive staged cells starting at
// row (shared memory); visibility v's first tap is at dxo[v] (= dx ov).  The
// table address is tab_adj + (bits of floor(t) + 2^23) * 8.  Accumulates
// P = sum A G' and Q = sum A dxo G' per visibility.
template <int kV>
__device__ __forceinline__ void row_taps(const float2 *__restrict__ row, int n, float (&dxo)[kV],
                                         const float (&dyo2)[kV], float ov, unsigned tab_adj, float (&pr)[kV],
                                         float (&pi)[kV], float (&qr)[kV], float (&qi)[kV]) {
    constexpr int kUnroll = 4;
#pragma unroll kUnroll
    for (int k = 0; k < n; ++k) {
        const float2 g = row[k];
#pragma unroll
        for (int v = 0; v < kV; ++v) {
            const float s2 = fmaf(dxo[v], dxo[v], dyo2[v]);
            const float t = sqrt_fast(s2);
            const float tf = __fadd_rz(t, 8388608.0f);          // floor(t) + 2^23
            const float2 e = lds_f2(tab_adj + ((unsigned)__float_as_int(tf) << 3));
            const float A = fmaf(t, e.y, e.x);
            fma2_acc(pr[v], pi[v], A, g.x, g.y);
            fma2_acc(qr[v], qi[v], __fmul_rn(A, dxo[v]), g.x, g.y);
            dxo[v] = __fsub_rn(dxo[v], ov);
        }
    }
}

// row_taps on staged w-planes: visibility v's cells start at lo[v] in its lower plane
// and `next` cells further in the upper one, whose weight is wf[v].
template <int kV>
__device__ __forceinline__ void row_taps_w(const float2 *const (&lo)[kV], int next, int n, float (&dxo)[kV],
                                           const float (&dyo2)[kV], const float (&wf)[kV], float ov, unsigned tab_adj,
                                           float (&pr)[kV], float (&pi)[kV], float (&qr)[kV], float (&qi)[kV]) {
#pragma unroll 4
    for (int k = 0; k < n; ++k) {
#pragma unroll
        for (int v = 0; v < kV; ++v) {
            const float2 g0 = lo[v][k], g1 = lo[v][next + k];
            const float2 g = ffma2(make_float2(wf[v], wf[v]), g1, ffma2(make_float2(-wf[v], -wf[v]), g0, g0));
            const float s2 = fmaf(dxo[v], dxo[v], dyo2[v]);
            const float t = sqrt_fast(s2);
            const float tf = __fadd_rz(t, 8388608.0f);          // floor(t) + 2^23
            const float2 e = lds_f2(tab_adj + ((unsigned)__float_as_int(tf) << 3));
            const float A = fmaf(t, e.y, e.x);
            fma2_acc(pr[v], pi[v], A, g.x, g.y);
            fma2_acc(qr[v], qi[v], A * dxo[v], g.x, g.y);
            dxo[v] -= ov;
        }
    }
}

}  // namespace tap
}  // namespace psc
