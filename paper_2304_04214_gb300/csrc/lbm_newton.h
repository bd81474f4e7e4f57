// lbm_newton.h -- the FP64 solve of eq:u_tau_implicit for the rare wall cell that
// FP32 does not settle.  Compiles as device code and, for checks, as plain C++.
#pragma once
#include <math.h>

#ifdef __CUDACC__
#define LBMK_DEVICE __device__ __forceinline__
#define LBMK_LOOP _Pragma("unroll 1")
#else
#define LBMK_DEVICE inline
#define LBMK_LOOP
#endif

namespace lbmk {

// e^-x, x >= 0, and p = 1 - e^-x: Taylor series of x / 2^n < 1/4, squared n times; p
// comes from the series itself where n = 0, so that both are good to a few times their
// last place below x = 1, and to 2^n of it beyond.  log(1 + z), z >= 0: two Halley steps on
// e^y = 1 + z from the FP32 logarithm, the residual z e^-y - p without cancellation near
// 0; error below 1e-14 of itself.  Loops instead of the unrolled library functions, whose
// code and registers weighed on every wall block.
LBMK_DEVICE double exp_neg_d(double x, double &p) {
    p = 1.0;
    if (x > 700.0) return 0.0;
    int n = 0;
    LBMK_LOOP
    while (x >= 0.25) { x *= 0.5; ++n; }
    double t = 1.0;
    LBMK_LOOP
    for (int k = 12; k > 1; --k) t = 1.0 - t * x * (1.0 / k);
    p = x * t;
    t = 1.0 - p;
    if (n == 0) return t;
    LBMK_LOOP
    for (; n > 0; --n) t *= t;
    p = 1.0 - t;
    return t;
}
LBMK_DEVICE double log1p_d(double z) {
    double y = (double)log1pf((float)z);
    LBMK_LOOP
    for (int it = 0; it < 2; ++it) {
        double p;
        const double e = exp_neg_d(y, p), d = fma(z, e, -p);     // (1 + z) / e^y - 1
        y += 2.0 * d / (2.0 + d);
    }
    return y;
}

LBMK_DEVICE float solve_utau_d(float uhat, float y1_nu, float kap, float B, float guess, bool *ok) {
    double u = guess;
    LBMK_LOOP
    for (int it = 0; it < 40; ++it) {
        const double yp = (double)y1_nu * u, k = kap;
        double p11, p3;
        const double e11 = exp_neg_d(yp * (1.0 / 11.0), p11), e3 = exp_neg_d(yp * (1.0 / 3.0), p3);
        const double up = log1p_d(k * yp) / k + B * (p11 - yp * (1.0 / 11.0) * e3);
        const double dup = 1.0 / (1.0 + k * yp) + B * ((e11 - e3) * (1.0 / 11.0) + yp * (1.0 / 33.0) * e3);
        const double du = (u * up - uhat) / (up + yp * dup);
        double un = u - du;
        if (!(un > 0.0)) un = 0.5 * u;
        u = un;
        if (fabs(du) <= 1e-12 * u) { *ok = true; return (float)u; }
    }
    *ok = false;
    return (float)u;
}

}  // namespace lbmk
