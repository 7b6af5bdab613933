// f64math.cuh -- FP64 reciprocals, square roots and the penalty norm in few
// FP64 instructions.
//
// GB300 issues one FP64 warp instruction per SM about every 16 cycles (1.2
// TFLOP/s measured against 74 in FP32), so FP64 code is bound by its number
// of FP64 instructions.  Reciprocals and inverse square roots start from an
// FP32 approximation of the mantissa (special-function unit, no FP64
// instruction; the exponent is integer work) and take one third-order
// Householder step, y (1 + e + e^2) and y (1 + e/2 + 3 e^2/8) with e the
// residual of the seed y, |e| < 1e-6: the truncation is below 1e-18 and the
// last multiply-add rounds once, so these are within one unit in the last
// place (0.51); a square root, x times the rounded inverse root, rounds a second
// time and is within two (1.6).  The largest eigenvalue of
// the penalty matrix starts from the FP32 polynomial of pair2.cuh and takes
// two Newton steps on 4 w^3 - 3 w = r.
// Arguments outside the plain range (zero, subnormal, infinite, NaN, very
// large or small) take the ordinary operations.
#pragma once
#include "dg_device.cuh"

namespace dg {

__device__ __forceinline__ float rcp_seed(float x)
{
    float r;
    asm("rcp.approx.ftz.f32 %0, %1;" : "=f"(r) : "f"(x));
    return r;
}
__device__ __forceinline__ float rsqrt_seed(float x)
{
    float r;
    asm("rsqrt.approx.ftz.f32 %0, %1;" : "=f"(r) : "f"(x));
    return r;
}

// the FP32 value f (normal, positive) times 2^n, as FP64, with sign bit `sign`
__device__ __forceinline__ double scaled_f64(float f, int n, unsigned sign)
{
    const unsigned b = __float_as_uint(f);
    const unsigned hi = sign | ((((b >> 23) + 896u) + static_cast<unsigned>(n)) << 20) | ((b & 0x7fffffu) >> 3);
    return __hiloint2double(static_cast<int>(hi), static_cast<int>(b << 29));
}

// 1 / x
__device__ __forceinline__ double rcp64(double x)
{
    const unsigned hi = static_cast<unsigned>(__double2hiint(x)), lo = static_cast<unsigned>(__double2loint(x));
    const unsigned ex = (hi >> 20) & 0x7ffu;
    if (ex - 64u > 1918u) return 1.0 / x;                 // |x| outside [2^-959, 2^959]
    const float m = __uint_as_float(0x3f800000u | ((hi & 0xfffffu) << 3) | (lo >> 29));
    const double y = scaled_f64(rcp_seed(m), 1023 - static_cast<int>(ex), hi & 0x80000000u);
    const double e = fma(-x, y, 1.0);
    return fma(y, fma(e, e, e), y);
}

// 1 / sqrt(x)
__device__ __forceinline__ double rsqrt64(double x)
{
    const unsigned hi = static_cast<unsigned>(__double2hiint(x)), lo = static_cast<unsigned>(__double2loint(x));
    const unsigned ex = hi >> 20;                          // sign and exponent: a negative x fails the test
    if (ex - 64u > 1918u) return 1.0 / sqrt(x);
    const int e2 = (static_cast<int>(ex) - 1023) & ~1;     // x = m 2^e2, m in [1, 4)
    const float m = __uint_as_float(((ex - 1023u - static_cast<unsigned>(e2) + 127u) << 23) |
                                    ((hi & 0xfffffu) << 3) | (lo >> 29));
    const double y = scaled_f64(rsqrt_seed(m), -(e2 / 2), 0u);
    const double e = fma(-x, y * y, 1.0);
    return fma(y, e * fma(0.375, e, 0.5), y);
}

// sqrt(x) for x >= 0
__device__ __forceinline__ double sqrt64(double x)
{
    const unsigned ex = static_cast<unsigned>(__double2hiint(x)) >> 20;
    if (ex - 64u > 1918u) return sqrt(x);
    return x * rsqrt64(x);
}

// cos(acos(r) / 3) in FP32 (the polynomial of sym3_max_eig2 in pair2.cuh)
__device__ __forceinline__ float third_angle_seed(float r)
{
    const float w = sqrtf(fminf(fmaxf(fmaf(0.5f, r, 0.5f), 0.0f), 1.0f));
    float c = fmaf(0.0011276363f, w, -0.0060893456f);
    c = fmaf(c, w, 0.016047280f);
    c = fmaf(c, w, -0.030235397f);
    c = fmaf(c, w, 0.052841410f);
    c = fmaf(c, w, -0.11103851f);
    c = fmaf(c, w, 0.57734692f);
    return fmaf(c, w, 0.5f);
}

// penalty_norm (dg_device.cuh) from (1 / rho, v1, v2, e): about 70 FP64
// instructions instead of 200.  w = cos(acos(r) / 3) is the largest root of
// 4 w^3 - 3 w = r; each Newton step forms its residual in FP64 and divides by
// the slope in FP32.  Near the double root (w = 1/2: the two largest
// eigenvalues meet) the slope vanishes, and the arccosine is taken.
__device__ __forceinline__ double penalty_norm64(double irho, double v1, double v2, double e, double n1, double n2,
                                                 const Phys<double> &ph)
{
    const double g = ph.gPr;
    const double vn = v1 * n1 + v2 * n2, vt = v2 * n1 - v1 * n2, vsq = v1 * v1 + v2 * v2, vn2 = vn * vn;
    const double a41 = fma(-g, e - vsq, fma(-1.0 / 3.0, vn2, -vsq));
    const double c42 = (4.0 / 3.0 - g) * vn, c43 = (1.0 - g) * vt;
    const double s11 = fma(16.0 / 9.0, vn2, 16.0 / 9.0);
    const double s12 = (4.0 / 3.0) * vn * vt;
    const double s13 = (4.0 / 3.0) * fma(-vn, a41, c42);
    const double s22 = fma(vt, vt, 1.0);
    const double s23 = fma(-vt, a41, c43);
    const double s33 = fma(a41, a41, fma(c42, c42, fma(c43, c43, g * g)));
    const double q = (s11 + s22 + s33) * (1.0 / 3.0);
    const double b11 = s11 - q, b22 = s22 - q, b33 = s33 - q;
    const double h = fma(s23, s23, fma(s13, s13, s12 * s12));
    const double p2 = fma(b11, b11, fma(b22, b22, fma(b33, b33, 2.0 * h))) * (1.0 / 6.0);
    double lam;
    const unsigned ex = static_cast<unsigned>(__double2hiint(p2)) >> 20;
    if (ex - 523u > 1000u) {                    // p2 outside [2^-500, 2^500], or not a positive number
        lam = sym3_max_eig(s11, s12, s13, s22, s23, s33);
        return ph.mu * irho * sqrt(lam > 0.0 ? lam : 0.0);
    }
    const double ip = rsqrt64(p2);
    const double det = fma(b11, fma(b22, b33, -s23 * s23),
                           fma(s13, fma(s12, s23, -b22 * s13), -s12 * fma(s12, b33, -s23 * s13)));
    const double r = (0.5 * det) * (ip * ip * ip);
    const float c = third_angle_seed(cvt_d2f(r));
    double w;
    if (c > 0.505f) {
        w = cvt_f2d(c);
        const float is = 1.0f / fmaf(12.0f * c, c, -3.0f);
#pragma unroll
        for (int it = 0; it < 2; ++it) {
            const double res = fma(w, fma(4.0 * w, w, -3.0), -r);
            w -= cvt_f2d(cvt_d2f(res) * is);
        }
    } else {
        w = cos(acos(fmin(fmax(r, -1.0), 1.0)) * (1.0 / 3.0));
    }
    lam = fma(2.0 * (p2 * ip), w, q);
    return ph.mu * irho * sqrt64(lam);
}

}  // namespace dg
