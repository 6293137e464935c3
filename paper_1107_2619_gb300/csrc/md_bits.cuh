// Conversions and scalings of FP64 values by their IEEE bit fields, in integer registers: GB300's
// FP64 pipe takes about 19 SM cycles per warp instruction whatever the number of active lanes
// (measured: 1.06 TFLOP/s of FMAs over 152 SMs), and it also executes the conversion instructions.
#pragma once

#include <cuda_runtime.h>
#include <string.h>

namespace mdk {
namespace eam {

// Conversions between FP64 and FP32: the exponent is
// rebiased by 1023 - 127 = 896 and the significand shifted by 29 bits.  f32_trunc: x >= 0 below
// the FP32 overflow threshold, rounded toward zero (relative error < 2^-23), and 0 below the
// normal FP32 range (so that coincident atoms still give 1/sqrt(0) = inf); f64_exact: f positive,
// normal or +inf, exact.
__device__ __forceinline__ float f32_trunc(double x) {
    const unsigned hi = (unsigned)__double2hiint(x), lo = (unsigned)__double2loint(x);
    return __uint_as_float(hi < (897u << 20) ? 0u : ((hi - (896u << 20)) << 3) | (lo >> 29));
}
__device__ __forceinline__ double f64_exact(float f) {
    const unsigned b = __float_as_uint(f);
    return b >= 0x7f800000u ? __hiloint2double(0x7ff00000, 0)
                            : __hiloint2double((int)((b >> 3) + (896u << 20)), (int)(b << 29));
}

// The rest x - f32_trunc(x) of a positive normal x, as FP32: its 29 low significand bits m, worth
// m 2^(E - 52), rounded to nearest (0 where m = 0 or E < -70, below which the exponent field
// would not hold it; the FP64 path's r^2 lie far inside).
__device__ __forceinline__ float f32_rest(double x) {
    const unsigned hi = (unsigned)__double2hiint(x), lo = (unsigned)__double2loint(x);
    const unsigned m = lo & 0x1FFFFFFFu;
    const int E = (int)(hi >> 20) - 1023;
    const float mf = __uint2float_rn(m);
    return (m == 0u || E < -70) ? 0.f : __int_as_float(__float_as_int(mf) + (E - 52) * (1 << 23));
}
// f as a double, exact, any sign: 0 for |f| below the normal FP32 range, NaN for inf or NaN.
__device__ __forceinline__ double f64_of_f32(float f) {
    const unsigned b = __float_as_uint(f), mag = b & 0x7fffffffu;
    const double v = __hiloint2double((int)((b & 0x80000000u) | ((mag >> 3) + (896u << 20))), (int)(mag << 29));
    return mag >= 0x7f800000u ? __hiloint2double(0x7ff80000, 0) : (mag < 0x00800000u ? 0.0 : v);
}

// x as FP32, rounded to nearest even as the conversion instruction does: 0 (signed) below FP32's
// normal range, infinity above it, NaN for NaN.
__device__ __forceinline__ float f32_rn(double x) {
    const unsigned hi = (unsigned)__double2hiint(x), lo = (unsigned)__double2loint(x);
    const unsigned mag = hi & 0x7fffffffu, sgn = hi & 0x80000000u;
    unsigned m = ((mag - (896u << 20)) << 3) | (lo >> 29);   // exponent and significand, truncated
    const unsigned rest = lo << 3;                            // the 29 bits below, half = 2^31
    m += (rest > 0x80000000u || (rest == 0x80000000u && (m & 1u))) ? 1u : 0u;   // a carry moves the exponent up
    if (mag < (897u << 20)) m = 0u;
    if (mag >= (1151u << 20)) m = (mag > 0x7ff00000u || (mag == 0x7ff00000u && lo)) ? 0x7fc00000u : 0x7f800000u;
    return __uint_as_float(sgn | m);
}
// x in units of 2^-fb as a whole number, rounded to nearest (0 <= fb <= 60), saturated to 62 bits.
__host__ __device__ __forceinline__ long long fix64(double x, int fb) {
#ifdef __CUDA_ARCH__
    const long long b = __double_as_longlong(x);
#else
    long long b;
    memcpy(&b, &x, sizeof b);
#endif
    const int e = (int)((b >> 52) & 0x7ff) - 1023;
    const long long m = (b & 0xFFFFFFFFFFFFFLL) | 0x10000000000000LL;
    const int s = e - 52 + fb;   // x = m 2^(e - 52)
    long long v;
    if (s >= 0) v = s <= 9 ? m << s : (1LL << 62);
    else v = s > -54 ? (m + (1LL << (-s - 1))) >> -s : 0;
    return b < 0 ? -v : v;
}

// Whether v is finite.
__device__ __forceinline__ bool finite64(double v) {
    return ((unsigned)__double2hiint(v) & 0x7ff00000u) != 0x7ff00000u;
}

// v / 2 by the exponent field (no FP64 operation); |v| below 2^-1021 (a subnormal half) gives 0.
__device__ __forceinline__ double half64(double v) {
    const long long b = __double_as_longlong(v);
    return (b & 0x7FF0000000000000LL) > (1LL << 52) ? __longlong_as_double(b - (1LL << 52)) : 0.0;
}
}  // namespace eam
}  // namespace mdk
