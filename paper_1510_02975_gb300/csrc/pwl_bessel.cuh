// pwl_bessel.cuh -- J0 and J1 for the Bessel test function f = A J0(alpha x)
// (Section V) and its second derivative A alpha^2 (J1(z)/z - J0(z)).
//
// Below x = 8 the CUDA library functions are used (their absolute error
// there is ~5e-16 in FP64).  From x = 8 on, the library's FP64 error grows
// to ~1e-13 (J0) and ~4e-13 (J1) by x = 250, which the density |f''|^{2/5}
// turns into knot errors above 1e-12 (b - a) for J0(alpha x) with
// alpha >= 3 on [0, 50].  There the modulus-phase form (DLMF 10.17)
//     J_nu(x) = sqrt(2 / (pi x)) (P_nu(x) cos chi - Q_nu(x) sin chi),
//     chi = x - (2 nu + 1) pi / 4,
// is evaluated with polynomials of P_nu and (x/8) Q_nu in u = (8/x)^2
// (pwl_bessel_tables.cuh, from gen_bessel_pq.py; one FP64 operation per term,
// where Clenshaw's sum of the same polynomial takes two: the FP64 pipe bounds
// every user of these functions), and with
//     cos chi0 = (cos x + sin x) / sqrt 2,   sin chi0 = (sin x - cos x) / sqrt 2,
//     cos chi1 = (sin x - cos x) / sqrt 2,   sin chi1 = -(sin x + cos x) / sqrt 2:
// absolute error ~3e-16.
#pragma once

#include <math.h>

#include "pwl_bessel_tables.cuh"

namespace pwl {

// c_0 + c_1 u + ... + c_{N-1} u^{N-1}
template <int N>
__device__ __forceinline__ double polynomial(const double* c, double u)
{
    double r = c[N - 1];
#pragma unroll
    for (int j = N - 2; j >= 0; --j) r = fma(r, u, c[j]);
    return r;
}

__device__ __forceinline__ double bessel_j0(double x)
{
    const double ax = fabs(x);
    if (ax < 8.0) return j0(x);
    const double t = 8.0 / ax, u = t * t;
    const double p = polynomial<16>(kBesselP0, u);
    const double q = t * polynomial<16>(kBesselQ0, u);
    double s, c;
    sincos(ax, &s, &c);
    return (p * (c + s) - q * (s - c)) * rsqrt(3.14159265358979323846 * ax);
}

__device__ __forceinline__ double bessel_j1(double x)
{
    const double ax = fabs(x);
    if (ax < 8.0) return j1(x);
    const double t = 8.0 / ax, u = t * t;
    const double p = polynomial<16>(kBesselP1, u);
    const double q = t * polynomial<16>(kBesselQ1, u);
    double s, c;
    sincos(ax, &s, &c);
    const double r = (p * (s - c) + q * (s + c)) * rsqrt(3.14159265358979323846 * ax);
    return x < 0.0 ? -r : r;
}

// FP32 (the FP32 design mode): the library's j0f / j1f (absolute error
// ~5e-7), within the FP32 mode's knot bound.
__device__ __forceinline__ float bessel_j0(float x) { return j0f(x); }
__device__ __forceinline__ float bessel_j1(float x) { return j1f(x); }

// J0(x) and J1(x)/x (f'' needs both; 1/2 - x^2/16 near 0): one sincos and one
// square root for the two, and 1/x = t/8.
__device__ __forceinline__ void bessel_j0_j1x(double x, double& j0v, double& j1x)
{
    const double ax = fabs(x);
    if (ax < 8.0) {
        j0v = j0(x);
        j1x = ax < 1e-8 ? 0.5 - x * x / 16.0 : j1(x) / x;
        return;
    }
    const double t = 8.0 / ax, u = t * t;
    const double p0 = polynomial<16>(kBesselP0, u), q0 = t * polynomial<16>(kBesselQ0, u);
    const double p1 = polynomial<16>(kBesselP1, u), q1 = t * polynomial<16>(kBesselQ1, u);
    double s, c;
    sincos(ax, &s, &c);
    const double r = rsqrt(3.14159265358979323846 * ax);
    j0v = (p0 * (c + s) - q0 * (s - c)) * r;
    j1x = (p1 * (s - c) + q1 * (s + c)) * r * (0.125 * t);
}

__device__ __forceinline__ void bessel_j0_j1x(float x, float& j0v, float& j1x)
{
    j0v = j0f(x);
    j1x = fabsf(x) < 1e-8f ? 0.5f - x * x / 16.0f : j1f(x) / x;
}

// J0 and J1 at the same point, FP32
__device__ __forceinline__ void bessel_j01(float x, float& j0v, float& j1v)
{
    j0v = j0f(x);
    j1v = j1f(x);
}

}  // namespace pwl
