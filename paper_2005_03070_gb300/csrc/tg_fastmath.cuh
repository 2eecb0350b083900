// Square root, its inverse and the reciprocal in few float64 instructions, for the serial chains of
// the small dense kernels: each is a seed and one cubic step,
//   1 / sqrt(x) = r (1 + e / 2 + 3/8 e^2),  e = 1 - x r^2   (Halley),
//   1 / x = r (1 + e + e^2),  e = 1 - x r.
// The seeds (rsqrt.approx.ftz.f64, rcp.approx.ftz.f64) are good to 2^-19, so that the steps leave less
// than 2^-55 and the last rounding: results are within 0.75 ulp.  sqrt_fast is within 1.25: its product x r
// is rounded once more, which costs the chains that use it one instruction less.  For x in mid_range.
#pragma once

namespace tg {

// 2^-900 <= x < 2^900, on the exponent bits
__device__ __forceinline__ bool mid_range(double x) {
    return (unsigned)((__double2hiint(x) >> 20) - 123) < 1800u;
}
__device__ __forceinline__ double rsqrt_seed(double x) {
    double r;
    asm("rsqrt.approx.ftz.f64 %0, %1;" : "=d"(r) : "d"(x));
    return r;
}
__device__ __forceinline__ double rsqrt_fast(double x) {
    const double r = rsqrt_seed(x), h = x * r, d = fma(x, r, -h), e = fma(-d, r, fma(-h, r, 1.0));    // d: what h lost
    return fma(r, e * fma(0.375, e, 0.5), r);
}
__device__ __forceinline__ double sqrt_fast(double x) {
    const double r = rsqrt_seed(x), h = x * r, e = fma(-h, r, 1.0);
    return fma(h * e, fma(0.375, e, 0.5), h);
}
__device__ __forceinline__ double rcp_seed(double x) {
    double r;
    asm("rcp.approx.ftz.f64 %0, %1;" : "=d"(r) : "d"(x));
    return r;
}
__device__ __forceinline__ double rcp_fast(double x) {
    const double r = rcp_seed(x), e = fma(-x, r, 1.0);
    return fma(r, fma(e, e, e), r);
}

}  // namespace tg
