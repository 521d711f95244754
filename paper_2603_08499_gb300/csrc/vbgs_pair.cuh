// vbgs_pair.cuh -- the logit of one (point, component) pair on the CUDA cores,
// shared by the dense passes (vbgs_estep_cc.cu) and the sparse ones
// (vbgs_estep_sparse.cu), and an exact FP32 -> FP64 conversion.
#pragma once
#include "vbgs_internal.cuh"

namespace vbgs {

__device__ __forceinline__ float ex2_approx(float x)
{
    float y;
    asm("ex2.approx.ftz.f32 %0, %1;" : "=f"(y) : "f"(x));
    return y;
}

template <typename T> struct Arith;
template <> struct Arith<double> {
    // r = exp(l - ref) in natural units
    static __device__ __forceinline__ double expd(double v) { return exp(v); }
    static __device__ __forceinline__ double lse_scale() { return 1.0; }
};
template <> struct Arith<float> {
    // records are in log2 units: r = 2^(l2 - ref2)
    static __device__ __forceinline__ float expd(float v) { return ex2_approx(v); }
    static __device__ __forceinline__ float lse_scale() { return 1.4426950408889634f; }
};

// logit (without the -psi(sum alpha) term) of point x under record r:
// c - 1/2 |M (x - m)|^2, M packed lower triangle at r[6..26].
template <typename T>
__device__ __forceinline__ T logit(const T *__restrict__ r, const T x[6])
{
    T d[6];
#pragma unroll
    for (int i = 0; i < 6; i++) d[i] = x[i] - r[i];
    T q = T(0);
#pragma unroll
    for (int i = 0; i < 6; i++) {
        T y = T(0);
#pragma unroll
        for (int j = 0; j <= i; j++) y = fma(r[6 + tri(i, j)], d[j], y);
        q = fma(y, y, q);
    }
    return fma(T(-0.5), q, r[27]);
}

// The first three rows (position only) of the same quadratic form, and the
// rest of it from there: the two halves together are logit's operations in
// logit's order.
__device__ __forceinline__ float quad_pos(const float *__restrict__ r, const float x[6])
{
    float d[3], q = 0.f;
#pragma unroll
    for (int i = 0; i < 3; i++) d[i] = x[i] - r[i];
#pragma unroll
    for (int i = 0; i < 3; i++) {
        float y = 0.f;
#pragma unroll
        for (int j = 0; j <= i; j++) y = fmaf(r[6 + tri(i, j)], d[j], y);
        q = fmaf(y, y, q);
    }
    return q;
}
__device__ __forceinline__ float quad_rest(const float *__restrict__ r, const float x[6], float q)
{
    float d[6];
#pragma unroll
    for (int i = 0; i < 6; i++) d[i] = x[i] - r[i];
#pragma unroll
    for (int i = 3; i < 6; i++) {
        float y = 0.f;
#pragma unroll
        for (int j = 0; j <= i; j++) y = fmaf(r[6 + tri(i, j)], d[j], y);
        q = fmaf(y, y, q);
    }
    return q;
}

// FP32 -> FP64 without an FP64 instruction: the exponent rebiased and the
// significand widened, exact for zeros and normal numbers; subnormals,
// infinities and NaNs take the conversion instruction.
__device__ __forceinline__ double f2d_exact(float f)
{
    const unsigned b = __float_as_uint(f);
    const unsigned ex = (b >> 23) & 0xffu;
    const unsigned long long sgn = (unsigned long long)(b & 0x80000000u) << 32;
    if ((b << 1) == 0u) return __longlong_as_double((long long)sgn);
    if (ex == 0u || ex == 0xffu) return (double)f;
    return __longlong_as_double((long long)(sgn | ((unsigned long long)(ex + 896u) << 52) |
                                            ((unsigned long long)(b & 0x7fffffu) << 29)));
}

// FP64 -> the pair h = RN32(v), l = RN32(v - h) without an FP64 instruction
// (each holds a warp's sub-partition for 64 cycles): the significand's top 24
// bits rounded to nearest even, and the signed remainder of at most 2^28
// units.  Zeros give (v, +0); values whose parts leave FP32's normal range
// take the conversions.
__device__ __forceinline__ void d2f_pair(double v, float &h, float &l)
{
    const unsigned long long b = (unsigned long long)__double_as_longlong(v);
    const int ex = (int)((b >> 52) & 0x7ff);
    if (ex < 949 || ex > 1149) {
        if ((b << 1) == 0ull) { h = __uint_as_float((unsigned)(b >> 32)); l = 0.f; return; }
        h = (float)v;
        l = (float)(v - (double)h);
        return;
    }
    const bool neg = (long long)b < 0;
    const unsigned top = (unsigned)((b >> 29) & 0x7fffffu) | 0x800000u, rem = (unsigned)b & 0x1fffffffu;
    const unsigned up = rem > 0x10000000u || (rem == 0x10000000u && (top & 1u)) ? 1u : 0u;
    const int hi = (int)(top + up), lo = (int)rem - (int)(up << 29);
    h = (float)(neg ? -hi : hi) * __uint_as_float((unsigned)(ex - 1046 + 127) << 23);
    l = (float)(neg ? -lo : lo) * __uint_as_float((unsigned)(ex - 1075 + 127) << 23);
}
} // namespace vbgs
