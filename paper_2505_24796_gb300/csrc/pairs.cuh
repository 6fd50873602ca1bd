// pairs.cuh -- two pixels a thread on CUDA cores: packed FP32 arithmetic, the Gaussian record it reads
// and the pixel layout, shared by the FP32 forward and the backward (render_fp32.cu).
#pragma once

#include "common.cuh"
#include "f32x2.cuh"

namespace tcgs {
namespace {

// x.lo y.lo + x.hi y.hi, the first product rounded.
__device__ __forceinline__ float dot2(f32x2 x, f32x2 y) { return fmaf(hi2(x), hi2(y), __fmul_rn(lo2(x), lo2(y))); }

// x where the half of `on` is not 0, else 0.
__device__ __forceinline__ f32x2 where2(f32x2 on, f32x2 x) {
    return pack2f(lo2(on) != 0.f ? lo2(x) : 0.f, hi2(on) != 0.f ? hi2(x) : 0.f);
}
constexpr float kHuge = 1e18f;   // magnitudes below this neither are nor make infinities in products of two

__device__ __forceinline__ float rcp_approx(float x) {
    float y;
    asm("rcp.approx.ftz.f32 %0, %1;" : "=f"(y) : "f"(x));
    return y;
}

// One level of a transposing butterfly over lanes that differ in `bit` (up: this lane has it set): the
// lower lane ends with the pair's sum of x, the upper one with that of y.
__device__ __forceinline__ float exchange(float x, float y, bool up, int bit) {
    const float send = up ? x : y, keep = up ? y : x;
    return keep + __shfl_xor_sync(0xffffffffu, send, bit);
}

// A Gaussian's values, each twice (as one operand of a packed instruction needs them).
struct __align__(16) PairRec {
    ulonglong2 q[5];   // {x, -a}, {-b, -c}, {y, -o}, {r, g}, {b, ln o}
    __device__ __forceinline__ float lno() const { return lo2(q[4].y); }
};

__device__ __forceinline__ PairRec pair_rec(float mx, float my, float a, float b, float c, float o, float r, float g,
                                            float bl, float lno) {
    PairRec v;
    v.q[0] = make_ulonglong2(pack2f(mx, mx), pack2f(-a, -a));
    v.q[1] = make_ulonglong2(pack2f(-b, -b), pack2f(-c, -c));
    v.q[2] = make_ulonglong2(pack2f(my, my), pack2f(-o, -o));
    v.q[3] = make_ulonglong2(pack2f(r, r), pack2f(g, g));
    v.q[4] = make_ulonglong2(pack2f(bl, bl), pack2f(lno, lno));
    return v;
}

// The exponent -(a dx^2 + c dy^2) / 2 - b dx dy from A = -a, B = -b, C = -c (Eq. 4); forward and backward
// take the same roundings, so a replay decides as the forward did.
__device__ __forceinline__ f32x2 pair_power(f32x2 A, f32x2 B, f32x2 C, f32x2 dx, f32x2 dy) {
    const f32x2 s = fma2(mul2(A, dx), dx, mul2(mul2(C, dy), dy));
    return fma2(s, pack2f(0.5f, 0.5f), mul2(mul2(B, dx), dy));
}

// A tile's 256 pixels over 128 threads: warp w owns the 8 x 8 block at (8 (w & 1), 8 (w >> 1)); lane l its
// pixels (lx, ly) and (lx, ly + 4).
constexpr int kPairThreads = 128;
struct PairPixels { int lx, ly; };
__device__ __forceinline__ PairPixels pair_pixels(int warp, int lane) {
    return PairPixels{8 * (warp & 1) + (lane & 7), 8 * (warp >> 1) + (lane >> 3)};
}

}  // namespace
}  // namespace tcgs
