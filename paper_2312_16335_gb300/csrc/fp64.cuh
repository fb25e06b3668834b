// FP64 reciprocals, roots and rotation angles for the eigenvalue kernels.
//
// FP64 on this chip: a warp instruction takes the pipe for 64 cycles, a division 550 and a root 585,
// and extra warps on a scheduler only queue.  So the kernels that use these keep one warp per scheduler,
// share no work redundantly between warps of a scheduler, and take reciprocals and roots from the
// hardware's approximations (about 2^-20 relative) by one cubic step:
//   1/x: y (1 + e + e^2), e = 1 - x y;   1/sqrt(x): y (1 + r/2 + 3 r^2/8), r = 1 - x y^2.
// The series leave out e^3, about 2^-60 relative.  What remains is rounding: the last fma (2^-53), and in the
// root x y before it (2^-54 of the result), so either is within 2^-52 of the exact value.  Against divisions and roots
// in the same places, on matrices of 5 to 768 rows, random, clustered and graded to 1e-12, the errors of eigenvalues,
// residuals and orthogonality (by 128-bit arithmetic) are the same or smaller.
#pragma once

#include <cuda_runtime.h>
#include <stdint.h>

namespace lv {

// 1 / x for 2^-1022 <= |x| <= 2^1021 (0 from about 2^1022 on, where the reciprocal is no normal number)
__device__ __forceinline__ double fast_rcp(double x) {
    double y;
    asm("rcp.approx.ftz.f64 %0, %1;" : "=d"(y) : "d"(x));
    const double e = fma(-x, y, 1.0);
    return fma(y, fma(e, e, e), y);
}
// 1 / sqrt(x) for a normal x > 0
__device__ __forceinline__ double fast_rsqrt(double x) {
    double y;
    asm("rsqrt.approx.ftz.f64 %0, %1;" : "=d"(y) : "d"(x));
    const double r = fma(-x * y, y, 1.0);
    return fma(y * r, fma(0.375, r, 0.5), y);
}

// v 2^-e as float32 (truncated; 0 below its range), e an exponent field >= v's: integer instructions only
__device__ __forceinline__ float scaled_float(double v, int e) {
    const int hi = __double2hiint(v), x = ((hi >> 20) & 0x7ff) - e + 127;
    const unsigned m = ((unsigned)hi & 0xfffffu) << 3 | (unsigned)__double2loint(v) >> 29;
    return x > 0 ? __uint_as_float(((unsigned)hi & 0x80000000u) | (unsigned)x << 23 | m) : 0.f;
}
// a float32 as FP64 (0 below its normal range), integer instructions only
__device__ __forceinline__ double float_bits_to_double(float f) {
    const unsigned u = __float_as_uint(f), x = (u >> 23) & 0xffu;
    if (x == 0u) return 0.0;
    return __hiloint2double((int)((u & 0x80000000u) | (x + 896u) << 20 | (u & 0x7fffffu) >> 3), (int)(u << 29));
}

// tangent t and cosine c of the rotation that (nearly) zeroes a_pq: rows p <- c (p - t q), q <- c (q + t p).  t is a
// float32 number (its error leaves 2^-21 of a_pq at most) and any t would do; c belongs to it in FP64, and it is
// the pair that has to be a rotation.  No rotation for |a_pq| below 2^-64 |a_qq - a_pp| either, where the square of
// theta is beyond float32.
__device__ __forceinline__ void jacobi_angle(double app, double aqq, double apq, double &t, double &c) {
    const double d = aqq - app;
    const int ed = (__double2hiint(d) >> 20) & 0x7ff, ex = (__double2hiint(apq) >> 20) & 0x7ff;
    const int e = max(ed, ex);
    const float theta = 0.5f * scaled_float(d, e) / scaled_float(apq, e);
    const float tf = copysignf(1.0f / (fabsf(theta) + sqrtf(fmaf(theta, theta, 1.0f))), theta);
    // no rotation for 0 / 0, a_pq below 2^-996 (about 1e-300) or entries that are not finite
    t = fabsf(tf) <= 1.0f && ex > 27 && e < 0x7ff ? float_bits_to_double(tf) : 0.0;
    const double u = fma(t, t, 1.0);
    double y;
    asm("rsqrt.approx.ftz.f64 %0, %1;" : "=d"(y) : "d"(u));  // about 2^-20
    const double r = fma(-u, y * y, 1.0);                     // y (1 + r / 2 + 3 r^2 / 8) is good to r^3
    c = fma(y * r, fma(0.375, r, 0.5), y);
}

}  // namespace lv
