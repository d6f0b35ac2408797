// What the walks over a tile's key list share (compositing, adjoint,
// importance): the staged record, the test which records of a batch can
// reach which 8x8 block of the tile, and packed FP32 pairs.
//
// A staged record is three float4s, 16 * kBatch bytes apart, so that one
// shared-memory offset addresses all of it:
//   [0] mean'x, mean'y, u00, u01   [1] u11, -log2 o', r, g
//   [2] b, -, pixel rect (x0 | y0 << 16, x1 | y1 << 16)
#pragma once

#include "common.cuh"

namespace lodge {

__device__ __forceinline__ void cp_async16(void* smem, const void* gmem) {
    unsigned s = (unsigned)__cvta_generic_to_shared(smem);
    asm volatile("cp.async.cg.shared.global [%0], [%1], 16;\n" ::"r"(s), "l"(gmem));
}
__device__ __forceinline__ void cp_async8(void* smem, const void* gmem) {
    unsigned s = (unsigned)__cvta_generic_to_shared(smem);
    asm volatile("cp.async.ca.shared.global [%0], [%1], 8;\n" ::"r"(s), "l"(gmem));
}
__device__ __forceinline__ void cp_async4(void* smem, const void* gmem) {
    unsigned s = (unsigned)__cvta_generic_to_shared(smem);
    asm volatile("cp.async.ca.shared.global [%0], [%1], 4;\n" ::"r"(s), "l"(gmem));
}
__device__ __forceinline__ void cp_async_commit() { asm volatile("cp.async.commit_group;\n" ::); }
__device__ __forceinline__ void cp_async_wait1() { asm volatile("cp.async.wait_group 1;\n" ::); }
__device__ __forceinline__ void cp_async_wait0() { asm volatile("cp.async.wait_group 0;\n" ::); }

// Two FP32 values in one 64-bit register pair: sm_103a issues their FMA,
// multiply and add as one instruction, each half rounded as the scalar form
// would be.
typedef unsigned long long f32x2;
__device__ __forceinline__ f32x2 pack2(float lo, float hi) {
    f32x2 r;
    asm("mov.b64 %0, {%1, %2};" : "=l"(r) : "f"(lo), "f"(hi));
    return r;
}
__device__ __forceinline__ void unpack2(f32x2 v, float& lo, float& hi) {
    asm("mov.b64 {%0, %1}, %2;" : "=f"(lo), "=f"(hi) : "l"(v));
}
__device__ __forceinline__ f32x2 fma2(f32x2 a, f32x2 b, f32x2 c) {
    f32x2 r;
    asm("fma.rn.f32x2 %0, %1, %2, %3;" : "=l"(r) : "l"(a), "l"(b), "l"(c));
    return r;
}
__device__ __forceinline__ f32x2 mul2(f32x2 a, f32x2 b) {
    f32x2 r;
    asm("mul.rn.f32x2 %0, %1, %2;" : "=l"(r) : "l"(a), "l"(b));
    return r;
}
// 1.0 where a >= b, else 0.0
__device__ __forceinline__ float ge01(float a, float b) {
    float r;
    asm("set.ge.f32.f32 %0, %1, %2;" : "=f"(r) : "f"(a), "f"(b));
    return r;
}

// Which of a tile's four 8x8 blocks (bit 0: top left, 1: top right, 2:
// bottom left, 3: bottom right; (tx0, ty0) the tile's first pixel) a record
// can reach with alpha >= 1/255 at a pixel centre.
//
// The record's tile rect must hold the tile (which the lists of coarser bins
// leave open), and its ellipse must reach the box of the block's pixel
// centres: with d = p - mean' and q(d) = (u00 dx + u01 dy)^2 + (u11 dy)^2 (the
// exponent's quadratic, a convex function with its minimum 0 at d = 0), the
// least q over the box [X, X + 7] x [Y, Y + 7] lies on dx = xc or on dy = yc,
// where xc, yc are the box coordinates nearest the mean (0 where the box
// spans it): along each line q is a one-dimensional quadratic whose minimiser
// (dy = -u00 u01 xc / (u01^2 + u11^2), dx = -u01 yc / u00) is clamped to the
// box.  A pixel centre can pass the 1/255 skip only if q <= log2 o' + log2
// 255 <= 8; the test adds a margin for the rounding of q, so it never drops a
// record that some pixel of the block would composite.  The covariance is at
// least 0.3 I, so that u00^2 and u01^2 + u11^2 are at most 2.41 and the terms
// of t and w at most M = 2.2 (max|dx| + max|dy|) over the tile; t and w, each
// a few roundings of them here and in the walk, differ by at most d = 11 eps M
// (eps = 2^-24), so that q differs by at most 2 sqrt(8) sqrt(2) d + 2 d^2 <=
// 5.3e-6 M + 9e-13 M^2.  With s = |dx| + |dy| at the tile's first pixel, M <=
// 2.2 (s + 30).  (s passes 1000 only where a splat of that many pixels reaches
// the tile from afar.  With a fixed margin of 0.01, one block in 3e5 lost a
// record of 3e5 pixels and one in ten one of 1e7.)
//
// One thread tests its record against all four blocks: the reciprocals are
// the record's, the clamped x terms a column's and the y terms a row's, so
// that four tests cost about 80 operations instead of 45 each.
//
// The record's pixel rect must meet the block as well: the rect holds the pixel
// centres within the extent, so a splat smaller than a pixel often misses a
// block that its ellipse, tested over the whole box of the centres, meets (four
// full-detail frames of 4M Gaussians 1540 us, 1575 with the ellipse alone).
// The rect's own rounding, 2^-23 of the coordinate, is within its margin of
// 0.05% of the extent but for splats of less than half a pixel far from the
// corner whose edge falls on a pixel centre within 2e-4 of a pixel.
//
// kKept (frames kept for the adjoint, the adjoint, scores) leaves nothing to
// that: the rect with a pixel around it counts (in the compositing of a lone
// chunk frame 64.1M warp instructions against 62.2M).  A record whose
// form is not a number (a covariance that overflows FP32) is kept there, as in
// a walk without the test; the plain frames drop it.
template <bool kKept>
__device__ __forceinline__ uint32_t blocks_met(const float4 a, const float4 b, const uint2 rect, uint32_t tx0,
                                               uint32_t ty0) {
    constexpr float kLog2_255 = 7.99435343f;
    const uint32_t rx0 = rect.x & 0xffffu, ry0 = rect.x >> 16, rx1 = rect.y & 0xffffu, ry1 = rect.y >> 16;
    if (rx0 > tx0 + 15u || rx1 < tx0 || ry0 > ty0 + 15u || ry1 < ty0) return 0u;
    constexpr uint32_t kGrow = kKept ? 1u : 0u;
    const bool cx[2] = {rx0 <= tx0 + 7u + kGrow, rx1 + kGrow >= tx0 + 8u};
    const bool cy[2] = {ry0 <= ty0 + 7u + kGrow, ry1 + kGrow >= ty0 + 8u};
    const float u00 = a.z, u01 = a.w, u11 = b.x;
    const float iy = __fdividef(-u00 * u01, fmaf(u01, u01, u11 * u11));
    const float ix = __fdividef(-u01, u00);
    float X0[2], X1[2], Y0[2], Y1[2], ym[2], ux[2], xm[2], uy[2], wy[2];
#pragma unroll
    for (int k = 0; k < 2; ++k) {
        X0[k] = (float)(tx0 + 8u * k) + 0.5f - a.x;
        X1[k] = X0[k] + 7.f;
        Y0[k] = (float)(ty0 + 8u * k) + 0.5f - a.y;
        Y1[k] = Y0[k] + 7.f;
        const float xc = fminf(fmaxf(0.f, X0[k]), X1[k]), yc = fminf(fmaxf(0.f, Y0[k]), Y1[k]);
        ym[k] = iy * xc;          // minimiser on the column's line dx = xc
        ux[k] = u00 * xc;
        xm[k] = ix * yc;          // minimiser on the row's line dy = yc
        uy[k] = u01 * yc;
        const float w = u11 * yc;
        wy[k] = w * w;
    }
    const float s = fabsf(X0[0]) + fabsf(Y0[0]);
    const float lim = fmaf(s, fmaf(5e-12f, s, 1.6e-5f), (kLog2_255 + 0.011f) - b.y);   // b.y = -log2 o'
    uint32_t met = 0;
#pragma unroll
    for (int r = 0; r < 2; ++r)
#pragma unroll
        for (int c = 0; c < 2; ++c) {
            const float dy = fminf(fmaxf(ym[c], Y0[r]), Y1[r]);
            const float t1 = fmaf(u01, dy, ux[c]), w1 = u11 * dy;
            const float dx = fminf(fmaxf(xm[r], X0[c]), X1[c]);
            const float t2 = fmaf(u00, dx, uy[r]);
            const float q = fminf(fmaf(t1, t1, w1 * w1), fmaf(t2, t2, wy[r]));
            if (cx[c] && cy[r] && (kKept ? !(q > lim) : q <= lim)) met |= 1u << (2 * r + c);
        }
    return met;
}

}  // namespace lodge
