// FP64 forms of the velocities and equilibria of lbrs_kernels.cuh with fewer FP64 operations and the
// same results (sm_103a).
//
// The FP64 path is bound by the chip's few FP64 units (about two operations per clock and SM), so an
// operation saved is time saved:
//  * both velocities share the reciprocal of rho: an approximate reciprocal refined by two steps, the
//    quotient q = m y corrected by its remainder, q' = q - (rho q - m) y.  With y the correctly rounded
//    reciprocal and an exact remainder, q' is the correctly rounded quotient (Markstein, "Computation of
//    elementary functions on the IBM RISC System/6000 processor", 1990), that is the IEEE division's,
//    with its sign also where it is zero (the remainder is then +0, and q - 0 is q).  Divisors and
//    dividends outside fp64_divisor_ok and fp64_quotient_ok take the division itself.  Unlike the
//    division's code it has no slow path for a zero momentum.
//  * U/4 and p's half are exact, so the product and the sum they go into may be fused.
// 1024^2 step: 160 us with two IEEE divisions and separate products (79 operations a cell without the
// divisions' own), 147 with the shared reciprocal by three Newton-Raphson steps, 141 with one cubic and
// one Newton-Raphson step and the momenta's zero tested on the integer units.
#pragma once

#include "lbrs_kernels.cuh"

namespace lbrs {

// The biased exponent lies in [256, 1790]: the size is between 2^-767 and 2^768.
__device__ __forceinline__ bool fp64_mid_range(double x)
{
    const unsigned e = ((unsigned)__double2hiint(x) >> 20) & 0x7ffu;
    return e - 256u <= 1790u - 256u;
}

// May x be divided by by its reciprocal?  It is positive and between 2^-250 and 2^251, so that a quotient of
// a mid-range dividend lies between 2^-1018 and 2^1018 (no overflow, no subnormal) and its remainder, a
// multiple of 2^-872 at least, is exact.  Not with a mantissa of all ones, whose reciprocal the last step
// may miss by one unit (1 - 2^-53: 1 instead of 1 + 2^-52).
__device__ __forceinline__ bool fp64_divisor_ok(double x)
{
    const unsigned hi = (unsigned)__double2hiint(x), lo = (unsigned)__double2loint(x);
    return (hi >> 20) - 773u <= 500u && (lo & (hi | 0xfff00000u)) != 0xffffffffu;
}

// 1/x, correctly rounded (fp64_divisor_ok).  The approximation reads and gives the upper word, within
// 2^-18; the hyperpower step of order three, y (1 + e + e^2) with e = 1 - x y (Altman, "An optimum cubically
// convergent iterative method of inverting a linear bounded operator in Hilbert space", 1960), leaves
// e^3 <= 2^-54 and its own rounding, within a unit in the last place; from there a Newton-Raphson step with
// an exact residual rounds correctly, but for a mantissa of all ones (Markstein).
__device__ __forceinline__ double fp64_reciprocal(double x)
{
    double y;
    asm("rcp.approx.ftz.f64 %0, %1;" : "=d"(y) : "d"(x));
    const double e = __fma_rn(-x, y, 1.0);
    y = __fma_rn(y, __fma_rn(e, e, e), y);
    return __fma_rn(y, __fma_rn(-x, y, 1.0), y);
}

// m / x from the reciprocal y of x.
__device__ __forceinline__ double fp64_quotient(double m, double x, double y)
{
    const double q = m * y;
    return __fma_rn(__fma_rn(x, q, -m), -y, q);
}

// The test for zero on the integer units: an FP64 comparison costs as much as a product.
__device__ __forceinline__ bool fp64_quotient_ok(double m)
{
    return fp64_mid_range(m) || (((unsigned)__double2hiint(m) << 1) | (unsigned)__double2loint(m)) == 0u;
}

// p / (gamma - 1) for many p: the reciprocal once.
struct Fp64Divisor {
    double x, y;
    bool ok;
    __device__ __forceinline__ explicit Fp64Divisor(double d) : x(d), y(0.0), ok(fp64_divisor_ok(d))
    {
        if (ok) y = fp64_reciprocal(d);
    }
    __device__ __forceinline__ double divide(double m) const
    {
        return ok && fp64_quotient_ok(m) ? fp64_quotient(m, x, y) : m / x;
    }
};

template <>
__device__ __forceinline__ void velocity2<double>(double rho, double mx, double my, double& u, double& v)
{
    if (fp64_divisor_ok(rho) && fp64_quotient_ok(mx) && fp64_quotient_ok(my)) {
        const double y = fp64_reciprocal(rho);
        u = fp64_quotient(mx, rho, y);
        v = fp64_quotient(my, rho, y);
    } else {
        u = mx / rho;
        v = my / rho;
    }
}

template <>
__device__ __forceinline__ double velocity1<double>(double rho, double m)
{
    if (fp64_divisor_ok(rho) && fp64_quotient_ok(m)) return fp64_quotient(m, rho, fp64_reciprocal(rho));
    return m / rho;
}

template <>
__device__ __forceinline__ void equilibria2d<double>(const double U[4], double gm1, double c, double e[4][4])
{
    double u, v;
    velocity2<double>(U[0], U[1], U[2], u, v);
    const double xx = U[1] * u, yy = U[2] * v;
    const double p = gm1 * __fma_rn(-0.5, xx + yy, U[3]), h = U[3] + p;
    const double F[4] = {U[1], xx + p, U[1] * v, u * h};
    const double G[4] = {U[2], U[2] * u, yy + p, v * h};
#pragma unroll
    for (int k = 0; k < 4; ++k) {
        const double b = c * F[k], d = c * G[k];
        const double am = __fma_rn(0.25, U[k], -b), ap = __fma_rn(0.25, U[k], b);
        e[0][k] = am - d;
        e[1][k] = ap - d;
        e[2][k] = ap + d;
        e[3][k] = am + d;
    }
}

template <>
__device__ __forceinline__ void equilibria1d<double>(const double U[3], double gm1, double c, double e[2][3])
{
    const double u = velocity1<double>(U[0], U[1]);
    const double xx = U[1] * u;
    const double p = gm1 * __fma_rn(-0.5, xx, U[2]);
    const double G[3] = {U[1], xx + p, u * (U[2] + p)};
#pragma unroll
    for (int k = 0; k < 3; ++k) {
        const double b = c * G[k];
        e[0][k] = __fma_rn(0.5, U[k], -b);
        e[1][k] = __fma_rn(0.5, U[k], b);
    }
}

// U/3 by the reciprocal's product and one correction, as above, at any size: a quotient by three lies at least
// a sixth of a unit in the last place from a tie, subnormal ones too, and the remainder is exact.  Not for
// infinities, whose product is the quotient and whose remainder is NaN.
__device__ __forceinline__ double fp64_third(double m)
{
    const double q = fp64_quotient(m, 3.0, 1.0 / 3.0);
    return ((unsigned)__double2hiint(m) & 0x7ff00000u) == 0x7ff00000u ? m : q;
}

template <>
__device__ __forceinline__ void equilibria1d3<double>(const double U[3], double gm1, double c, double e[3][3])
{
    const double u = velocity1<double>(U[0], U[1]);
    const double xx = U[1] * u;
    const double p = gm1 * __fma_rn(-0.5, xx, U[2]);
    const double G[3] = {U[1], xx + p, u * (U[2] + p)};
#pragma unroll
    for (int k = 0; k < 3; ++k) {
        const double a = fp64_third(U[k]);
        const double b = c * G[k];
        e[0][k] = a - b;
        e[1][k] = a;
        e[2][k] = a + b;
    }
}

// bound2d's local bound by one reciprocal of rho for its three quotients, the same bits (adaptive 768^2
// step 157 us with the three divisions, 141 so).
template <>
__device__ __forceinline__ double bound_local<double>(const double U[4], double gamma)
{
    if (!fp64_divisor_ok(U[0]) || !fp64_quotient_ok(U[1]) || !fp64_quotient_ok(U[2])) return bound2d<double>(U, gamma);
    const double gm1 = gamma - 1.0;
    const double y = fp64_reciprocal(U[0]);
    const double u = fp64_quotient(U[1], U[0], y), v = fp64_quotient(U[2], U[0], y);
    const double p = gm1 * __fma_rn(-0.5, U[1] * u + U[2] * v, U[3]);
    const double gp = gamma * p;
    if (!(U[0] > 0.0) || !(p > 0.0) || !isfinite(p)) return -1.0;
    const double a = sqrt(fp64_mid_range(gp) ? fp64_quotient(gp, U[0], y) : gp / U[0]);
    return fabs(u) + fabs(v) + sqrt(2.0) * a;
}

}  // namespace lbrs
