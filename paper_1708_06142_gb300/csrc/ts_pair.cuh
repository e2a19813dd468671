// FP32 helpers of the paired walks (two children per packed f32x2 instruction) shared by the gravity and
// the column walk.
#pragma once
#include <cuda_runtime.h>
#include <stdint.h>

// 1/sqrt(x).  SUB = false: the hardware instruction alone, which flushes subnormal inputs.  rsqrtf
// also rescales those, three more instructions on every call (24 of the ~200 of a popped group: the
// 2M-cell Plummer BH walk ran 9 % longer with it); it is kept for meshes whose cells are so small
// that a squared separation can be subnormal (WalkParams::tiny).  Normal inputs give the same bits.
template <bool SUB>
__device__ __forceinline__ float rsq(float x) {
    if constexpr (SUB) return rsqrtf(x);
    float y;
    asm("rsqrt.approx.ftz.f32 %0, %1;" : "=f"(y) : "f"(x));
    return y;
}
// 32-byte record by one 256-bit load.  Measured on GB300 with scattered addresses: a 128-bit load
// costs the L1 one cycle per distinct 128-byte line of the warp, a 256-bit load half a cycle per
// distinct line of each group of 4 lanes, so a record costs half or less of two 128-bit loads.
__device__ __forceinline__ void ld_rec(const float4* p, float4& a, float4& b) {
    asm("ld.global.nc.v8.f32 {%0, %1, %2, %3, %4, %5, %6, %7}, [%8];"
        : "=f"(a.x), "=f"(a.y), "=f"(a.z), "=f"(a.w), "=f"(b.x), "=f"(b.y), "=f"(b.z), "=f"(b.w)
        : "l"(p));
}

// Minimum image of two separations at once: d - L rint(d / L), the rounding to the nearest integer by
// adding and subtracting 1.5 * 2^23 (exact below 2^22; additions where rintf needs the conversion unit for
// each value).  An isolated axis has 1 / L = L = 0.  The product is rounded by itself, as in the scalar
// walks, so that a separation of exactly half a period keeps its sign whichever way 1 / L rounds: the first
// addition is scalar because a packed one is fused with the packed product, and then half the boxes flip
// such pairs (column maps off by up to 80 % in pixels facing them).  The two scalar additions cost 1.4 % of
// the 128^3 column walk (19.97 -> 20.25 ms) and 2.1 % of the 128^3 Taylor walk (15.6 -> 15.9 ms); a product with
// subnormals flushed, which is not fused either, 1.9 % and 1.6 %.
__device__ __forceinline__ float2 pk_image(float2 d, float2 iL, float2 nL) {
    const float2 q = __fmul2_rn(d, iL);
    const float2 r = make_float2(__fadd_rn(q.x, 12582912.f), __fadd_rn(q.y, 12582912.f));
    return __ffma2_rn(__fadd2_rn(r, make_float2(-12582912.f, -12582912.f)), nL, d);
}

// d^2 as the scalar kernels form it, fma(dx, dx, dy dy) + dz dz with the last product rounded by
// itself, so that every MAC decision is theirs bit for bit.  (The last addition is scalar: a packed
// one is fused with the packed product.)
__device__ __forceinline__ float2 pk_norm2(float2 dx, float2 dy, float2 dz) {
    const float2 a = __ffma2_rn(dx, dx, __fmul2_rn(dy, dy)), b = __fmul2_rn(dz, dz);
    return make_float2(__fadd_rn(a.x, b.x), __fadd_rn(a.y, b.y));
}
