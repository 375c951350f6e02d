// tcx_slices.cuh -- device helpers of the sliced BF16 number format (tcx_gemm.cuh): group
// exponents, the four slices of a two-float value, two-float sums and products.
#pragma once
#include <cuda_runtime.h>
#include <stdint.h>

namespace coro {

__device__ __forceinline__ float pow2f(int k) { return __int_as_float((k + 127) << 23); }   // k in [-126, 127]

// Exponent e of the smallest power of two >= |x| for x > 0 (normal).
__device__ __forceinline__ int ceil_log2(float ax) {
    const uint32_t b = __float_as_uint(ax);
    const int ex = (int)((b >> 23) & 0xff) - 127;
    return (b & 0x7fffff) ? ex + 1 : ex;
}

// Largest |value| of the warp's 32 lanes (all lanes must call), as float bits: non-negative
// floats order like their bit patterns.
__device__ __forceinline__ uint32_t warp_max_bits(float amax) {
    return __reduce_max_sync(0xffffffffu, __float_as_uint(amax));
}

// Group exponent from the group's largest magnitude m (float bits): 2^e >= every |value|.
// Clamped to [-90, 120] so that every slice scale 2^(e - 32) stays a normal float.
__device__ __forceinline__ int group_exp_of(uint32_t m) {
    if (m == 0) return -90;
    int e = ceil_log2(__uint_as_float(m));
    return e < -90 ? -90 : (e > 120 ? 120 : e);
}

// Exponent of a 64-element group held by two consecutive warps of a block (warps 2w, 2w + 1);
// every thread of the block calls (two block barriers). sh: one word per warp.
__device__ __forceinline__ int group64_exp_block(float amax, uint32_t* sh) {
    const uint32_t wm = warp_max_bits(amax);
    const int w = threadIdx.x >> 5;
    if ((threadIdx.x & 31) == 0) sh[w] = wm;
    __syncthreads();
    const uint32_t m = max(sh[w & ~1], sh[w | 1]);
    __syncthreads();
    return group_exp_of(m);
}

// Four slices of the two-float value (h, l) in the group with exponent e.
__device__ __forceinline__ void make_slices(float h, float l, int e, float (&s)[4]) {
    const float t = h * pow2f(8 - e), tl = l * pow2f(8 - e);
    const float a0 = rintf(t);
    float r = (t - a0) + tl;                           // t - a0 is exact
    s[0] = a0 * pow2f(e - 8);
    r *= 256.f;
    const float a1 = rintf(r);
    r -= a1;
    s[1] = a1 * pow2f(e - 16);
    r *= 256.f;
    const float a2 = rintf(r);
    r -= a2;
    s[2] = a2 * pow2f(e - 24);
    s[3] = rintf(r * 256.f) * pow2f(e - 32);
}

__device__ __forceinline__ void two_sum(float a, float b, float& s, float& err) {
    s = a + b;
    const float bb = s - a;
    err = (a - (s - bb)) + (b - bb);
}

// (h, l) * (sh, sl) -> normalised two-float product
__device__ __forceinline__ void mul22(float h, float l, float sh, float sl, float& ph, float& pl) {
    const float p = h * sh;
    float e = fmaf(h, sh, -p);
    e += h * sl + l * sh;
    ph = p + e;
    pl = e - (ph - p);
}

}  // namespace coro
