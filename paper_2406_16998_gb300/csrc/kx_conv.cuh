// Device helpers shared by the kernels: float64 <-> float32 conversions by integer
// operations, packed f32x2 arithmetic, split scales and fp16 hi / lo splits, and
// compensated sums.
#pragma once
#include <cuda_fp16.h>
#include <cuda_runtime.h>

namespace kx {

// Conversions between float64 and float32 with integer operations: on this
// GPU the hardware conversions run on the float64 pipe, which is slow enough
// that they, not memory, would bound the kernels that use them.  Finite values in the
// float32 normal range convert as IEEE rounding would, up to the tie rule
// (half-ulp ties round away from zero); magnitudes below 2^-126 become zero
// or a float32 subnormal below 2^-146, magnitudes beyond the float32 range a
// non-finite value.
__device__ __forceinline__ float f64_to_f32(double d) {
    const unsigned long long u = (unsigned long long)__double_as_longlong(d);
    const unsigned lo = (unsigned)u;
    unsigned hi = (unsigned)(u >> 32);
    const unsigned lo_r = lo + 0x10000000u;  // half of the last kept mantissa bit
    hi += (lo_r < lo) ? 1u : 0u;             // its carry
    // float64 exponent 896 + e is float32 exponent e: clamp to 0 .. 255, rebias
    const unsigned ax = min(max(hi & 0x7fffffffu, 896u << 20), 1151u << 20) - (896u << 20);
    return __uint_as_float((hi & 0x80000000u) | (ax << 3) | (lo_r >> 29));
}

__device__ __forceinline__ double f32_to_f64(float f) {
    const unsigned b = __float_as_uint(f);
    const unsigned sgn = b & 0x80000000u, ax = b & 0x7fffffffu;
    unsigned hi = sgn, lo = 0u;
    if (ax >= 0x7f800000u) {
        hi = sgn | 0x7ff00000u;
    } else if (ax >= 0x00800000u) {
        hi = sgn | ((ax >> 3) + (896u << 20));
        lo = ax << 29;
    }
    return __hiloint2double((int)hi, (int)lo);
}

// s += a * b on both lanes of a float pair, one packed instruction.
__device__ __forceinline__ void fma2(float2 &s, float2 a, float2 b) {
    unsigned long long rs = *reinterpret_cast<unsigned long long *>(&s);
    asm("fma.rn.f32x2 %0, %1, %2, %0;"
        : "+l"(rs)
        : "l"(*reinterpret_cast<unsigned long long *>(&a)), "l"(*reinterpret_cast<unsigned long long *>(&b)));
    s = *reinterpret_cast<float2 *>(&rs);
}

// Split scales: powers of two from an item's maximum.
__device__ __forceinline__ int scale_exp(float mx) {
    // e such that mx * 2^e < 2^14 (mx = m 2^k, m in [0.5, 1)  =>  e = 14 - k), from the
    // exponent bits (frexpf only for subnormal maxima)
    int k = 0;
    if (mx > 0.f && isfinite(mx)) {
        k = (__float_as_int(mx) >> 23) - 126;
        if (k == -126) frexpf(mx, &k);
    }
    return 14 - k;
}
__device__ __forceinline__ float pow2f(int e) {
    return (unsigned)(e + 126) < 254u ? __int_as_float((e + 127) << 23) : ldexpf(1.f, e);
}

// Packed float32 arithmetic (two values per instruction, each rounded as the scalar
// form rounds it): the tensor-core kernels' epilogues and producers are bound by the
// length of their instruction sequences.
__device__ __forceinline__ float2 add2(float2 a, float2 b) {
    unsigned long long r;
    asm("add.rn.f32x2 %0, %1, %2;"
        : "=l"(r)
        : "l"(*reinterpret_cast<unsigned long long *>(&a)), "l"(*reinterpret_cast<unsigned long long *>(&b)));
    return *reinterpret_cast<float2 *>(&r);
}
__device__ __forceinline__ float2 mul2(float2 a, float2 b) {
    unsigned long long r;
    asm("mul.rn.f32x2 %0, %1, %2;"
        : "=l"(r)
        : "l"(*reinterpret_cast<unsigned long long *>(&a)), "l"(*reinterpret_cast<unsigned long long *>(&b)));
    return *reinterpret_cast<float2 *>(&r);
}

// Eight values into their fp16 hi and lo parts, 16 bytes each.
__device__ __forceinline__ void split8(const float2 *v, uint4 &hi, uint4 &lo) {
    __half2 h[4], l[4];
#pragma unroll
    for (int i = 0; i < 4; ++i) {
        const __half2 hh = __floats2half2_rn(v[i].x, v[i].y);
        float2 r = v[i];
        fma2(r, __half22float2(hh), make_float2(-1.f, -1.f));
        h[i] = hh;
        l[i] = __floats2half2_rn(r.x, r.y);
    }
    hi = *reinterpret_cast<uint4 *>(h);
    lo = *reinterpret_cast<uint4 *>(l);
}

__device__ __forceinline__ float2 pair(const float *v, int k) { return make_float2(v[2 * k], v[2 * k + 1]); }

// (hi, lo) += v with the rounding error of the float32 addition kept in lo.
__device__ __forceinline__ void two_sum_add(float &hi, float &lo, float v) {
    const float t = hi + v;
    const float bp = t - hi;
    lo += (hi - (t - bp)) + (v - bp);
    hi = t;
}

}  // namespace kx
