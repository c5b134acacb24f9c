// fp64_dev.cuh -- FP64 roots and quotients for kernels that the FP64 pipe
// bounds (1/73 of the FP32 rate on this GPU): Newton iterations from an FP32
// seed, and FP32 inputs widened by their bits.
#pragma once
#include <cstdint>

namespace pic {

// a float as a double, by its bits (zero, denormals, infinities and NaN by
// the conversion)
__device__ __forceinline__ double widen(float f)
{
    const uint32_t b = __float_as_uint(f), e = (b >> 23) & 0xffu;
    if (e - 1u >= 254u) return (double)f;
    return __hiloint2double((int)((b & 0x80000000u) | (((b & 0x7fffffffu) >> 3) + 0x38000000u)), (int)(b << 29));
}
__device__ __forceinline__ double widen(double f) { return f; }

// 1/sqrt(a) for a >= 1: the FP32 root of a's leading bits, then two Newton
// steps (7e-7 -> 7e-13 -> rounding); beyond FP32's range the library's root
__device__ __forceinline__ double rsqrt_fp64(double a)
{
    const uint32_t hi = (uint32_t)__double2hiint(a);
    if (hi >= 0x46000000u) return 1.0 / sqrt(a);  // a >= 2^97, infinity, NaN
    double r = widen(rsqrtf(__uint_as_float((hi - 0x38000000u) << 3)));
    const double h = 0.5 * a;
    r = fma(r, fma(-h, r * r, 0.5), r);
    return fma(r, fma(-h, r * r, 0.5), r);
}

// 1/b for b >= 1, the same way
__device__ __forceinline__ double rcp_fp64(double b)
{
    const uint32_t hi = (uint32_t)__double2hiint(b);
    if (hi >= 0x46000000u) return 1.0 / b;
    double q = widen(__frcp_rn(__uint_as_float((hi - 0x38000000u) << 3)));
    q = fma(q, fma(-b, q, 1.0), q);
    return fma(q, fma(-b, q, 1.0), q);
}

// the integer nearest to x (|x| < 2^31; of two, the even one) as a double and
// as an int, by adding and taking away 1.5 2^52
__device__ __forceinline__ double nearest_fp64(double x, int &i)
{
    const double t = x + 6755399441055744.0;
    i = __double2loint(t);
    return t - 6755399441055744.0;
}

}  // namespace pic
