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

// e^-x, x >= 0: Taylor series of e^(-x / 2^n), x / 2^n < 1/4, squared n times; its
// error is below 1e-15 of 1, relative to itself below 1e-12.  log(1 + z), z >= 0: a
// series below 0.05, else two Halley steps on e^y = 1 + z from the FP32 logarithm; error
// below 1e-14 of itself.  Loops instead of the unrolled library functions, whose code
// and registers weighed on every wall block.
LBMK_DEVICE double exp_neg_d(double x) {
    if (x > 700.0) return 0.0;
    int n = 0;
    LBMK_LOOP
    while (x >= 0.25) { x *= 0.5; ++n; }
    double t = 1.0;
    LBMK_LOOP
    for (int k = 12; k > 0; --k) t = 1.0 - t * x * (1.0 / k);
    LBMK_LOOP
    for (; n > 0; --n) t *= t;
    return t;
}
LBMK_DEVICE double log1p_d(double z) {
    if (z < 0.05) {
        double t = 0.0;
        LBMK_LOOP
        for (int k = 12; k > 0; --k) t = 1.0 / k - t * z;
        return z * t;
    }
    double y = (double)log1pf((float)z);
    LBMK_LOOP
    for (int it = 0; it < 2; ++it) {
        const double w = (1.0 + z) * exp_neg_d(y);     // (1 + z) / e^y
        y += 2.0 * (w - 1.0) / (w + 1.0);
    }
    return y;
}

LBMK_DEVICE float solve_utau_d(float uhat, float y1_nu, float kap, float B, float guess, bool *ok) {
    double u = guess;
    LBMK_LOOP
    for (int it = 0; it < 40; ++it) {
        const double yp = (double)y1_nu * u, k = kap;
        const double e11 = exp_neg_d(yp * (1.0 / 11.0)), e3 = exp_neg_d(yp * (1.0 / 3.0));
        const double up = log1p_d(k * yp) / k + B * (1.0 - e11 - yp * (1.0 / 11.0) * e3);
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
