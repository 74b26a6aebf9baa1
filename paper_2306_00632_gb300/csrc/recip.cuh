// Reciprocals from an estimate and one correction, for chains of dependent instructions.
//
// With r about 1/q and e = 1 - q r,  1/q = r / (1 - e) = r (1 + e + e^2 + e^3 + ...), the geometric series: cut after e^2 it
// is the third-order Newton (Householder) iteration, after e Newton's.  An FP32 estimate of q's leading 24 bits has
// |e| < 1e-6, so that the FP64 form cuts off less than 1e-18 and rounds once in its last FMA: within 1.05 u of 1/q (u = 2^-53).
// In the same way d^(-1/2) = y (1 - e)^(-1/2) = y (1 + e/2 + 3 e^2/8 + ...) with e = 1 - d y^2 (binomial series).
//
// Measured, with IEEE divisions in their place: the three FP64 Grams of a truncation of order 97 1675 us, so 1562; of
// order 32 638 us, so 564 (1.3% of it from the Cholesky's reciprocals, the rest from the rotations').
#pragma once

namespace tpcg {

// Conversions by moving bits (an FP64 conversion takes its quarter of an SM as long as any FP64 instruction of a warp, 64
// cycles): v 2^-off as a float (mantissa cut, not rounded; 0 below FP32's range), and a normal float as a double times 2^off
__device__ __forceinline__ float bits_to_float(double v, int off = 0) {
    const int hi = __double2hiint(v);
    const int e = ((hi >> 20) & 0x7ff) - (1023 - 127) - off;
    const int bits = (hi & 0x80000000) | (e << 23) | ((hi & 0xfffff) << 3) | ((unsigned)__double2loint(v) >> 29);
    return e > 0 ? __int_as_float(bits) : 0.f;
}
__device__ __forceinline__ double bits_to_double(float f, int off = 0) {
    const unsigned b = __float_as_uint(f);
    const int hi = (int)((b & 0x80000000u) | (((b & 0x7fffffffu) >> 3) + ((unsigned)(1023 - 127 + off) << 20)));
    return __hiloint2double(hi, (int)(b << 29));
}

// 1 / q from the estimate r (|1 - q r| < 1e-6)
__device__ __forceinline__ double recip_from(double q, double r) {
    const double e = fma(-q, r, 1.0);
    return fma(r, fma(e, e, e), r);
}
__device__ __forceinline__ float recip_from(float q, float r) { return fmaf(r, fmaf(-q, r, 1.f), r); }
// 1 / q for q from 2^-125 to 2^125
__device__ __forceinline__ double recip_mid(double q) {
    return recip_from(q, bits_to_double(__fdividef(1.f, bits_to_float(q))));
}
// d^(-1/2) from the estimate y: within 1.6 u (u = 2^-24)
__device__ __forceinline__ float rsqrt_from(float d, float y) { return fmaf(y * fmaf(-d * y, y, 1.f), 0.5f, y); }

}  // namespace tpcg
