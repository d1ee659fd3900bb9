// 1/sqrt(x), sqrt(x) and 1/q in FP64 from FP32 seeds, and the Jastrow term made of them.
//
// The sums over pairs wait for the FP64 pipe (a warp instruction every 16 cycles of an SM), so the
// seeds come from the FP32 reciprocal square root and reciprocal, and one third-order step each
// (Halley's for the root) makes them FP64.  Against 64 more bits, 4 million arguments, in units of
// the last place, mean / largest, beside correctly rounded sqrt and division:
//   1/sqrt(x)   0.250 / 0.500   (1 / sqrt: 0.355 / 1.49; CUDA's rsqrt documents 1)
//   U           0.528 / 3.1     (0.528 / 3.5)
//   U' / r      0.936 / 6.3     (0.992 / 6.8)
//   lap U       4.64            (5.40; its two terms cancel)
// (x y taken before its square instead of y^2 exactly, and r = x / sqrt(x) without its residual, left
// U at 0.554 and lap U at 5.62.)
#pragma once

namespace qmc {

// 2^-99 <= x < 2^99, by its exponent (an FP64 compare goes through the FP64 pipe too)
__device__ __forceinline__ bool in_fast_range(double x)
{
    return (unsigned)__double2hiint(x) - 0x39c00000u < 0x0c600000u;
}

__device__ __forceinline__ double half_normal(double x)   // 0.5 x where x / 2 is a normal number
{
    return __hiloint2double(__double2hiint(x) - 0x00100000, __double2loint(x));
}

// From the FP32 reciprocal square root y (relative error 2^-22): with e = 1 - x y^2 (y^2 exact in
// FP64), 1/sqrt(x) = y (1 - e)^(-1/2) = y (1 + e/2 + 3 e^2/8 + O(e^3)), O(e^3) < 2^-64.
__device__ __forceinline__ double rsqrt_f64(double x)
{
    if (!in_fast_range(x)) return rsqrt(x);
    const double y = (double)rsqrtf((float)x);
    const double e = fma(-x, y * y, 1.0);
    return fma(e * y, fma(0.375, e, 0.5), y);
}

// One Jastrow term, Pade form U = a r / (1 + b r): U' = a / (1 + b r)^2, U'' = -2 a b / (1 + b r)^3,
// lap U(|r_e - x|) = U'' + 2 U' / r, grad U = U' (r_e - x) / r.  f = U' / r.
__device__ __forceinline__ void jastrow_term(double r2, double a, double b, double &f, double &lap, double &u)
{
    double iq, ir, r, q;
    bool fast = in_fast_range(r2);
    if (fast) {
        ir = rsqrt_f64(r2);
        r = r2 * ir;
        r = fma(fma(-r, r, r2), half_normal(ir), r);    // Heron's step from the residual: sqrt(r2)
        q = 1.0 + b * r;
        fast = in_fast_range(q);
    }
    if (fast) {
        // 1 / q from the FP32 reciprocal y: with e = 1 - q y, 1 / q = y (1 + e + e^2 + O(e^3))
        const double y = (double)__frcp_rn((float)q);
        const double e = fma(-q, y, 1.0);
        iq = fma(y, fma(e, e, e), y);
        const double t = a * iq;
        u = t * r;
        const double u1 = t * iq;
        f = u1 * ir;
        lap = fma(2.0, f, -2.0 * b * (u1 * iq));
    } else {
        r = sqrt(r2);
        q = 1.0 + b * r;
        iq = 1.0 / q;
        const double u1 = a * iq * iq;
        f = u1 / r;
        lap = -2.0 * a * b * iq * iq * iq + 2.0 * f;
        u = a * r * iq;
    }
}

}  // namespace qmc
