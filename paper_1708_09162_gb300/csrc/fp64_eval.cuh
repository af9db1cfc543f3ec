// FP64 evaluation of the fundamental solutions on the device.  GB300 issues 2 FP64
// operations per clock and SM, so every kernel that evaluates them in FP64 is
// bound by their count.
#pragma once

#include <cuda_runtime.h>

#include <cmath>
#include <vector>

namespace ibem {

// e^{i theta} from a table and Taylor series: theta = n c + t, c = 2 pi / 512,
// |t| <= c / 2, with c in two parts; e^{i n c} from the table of cos and sin,
// sin t = t - t^3/6 + t^5/120, cos t - 1 = -t^2/2 + t^4/24 - t^6/720 (the next terms
// are below 2^-56).  15 FP64 operations for both.
constexpr int TRIG64_N = 512;

// the table, [TRIG64_N] (cos, sin), computed in extended precision
inline std::vector<double> trig64_table() {
    std::vector<double> t(2 * TRIG64_N);
    const long double c = 6.283185307179586476925286766559005768L / TRIG64_N;
    for (int j = 0; j < TRIG64_N; ++j) {
        t[2 * j] = (double)std::cos(c * j);
        t[2 * j + 1] = (double)std::sin(c * j);
    }
    return t;
}

__device__ __forceinline__ void expi64(double theta, const double2* __restrict__ tab, double* cs, double* sn) {
    constexpr double pi = 3.14159265358979323846;
    constexpr double chi = 2.0 * pi / TRIG64_N;                        // c rounded
    constexpr double clo = 2.0 * 1.2246467991473532e-16 / TRIG64_N;    // pi minus its rounded value, scaled
    const double m = fma(theta, 1.0 / chi, 6755399441055744.0);        // + 1.5 2^52: n in the low bits
    const double n = m - 6755399441055744.0;
    const double t = fma(-n, clo, fma(-n, chi, theta));
    const double2 e = __ldg(tab + (__double2loint(m) & (TRIG64_N - 1)));
    const double t2 = t * t;
    const double st = fma(t * t2, fma(t2, 1.0 / 120.0, -1.0 / 6.0), t);
    const double ct = t2 * fma(t2, fma(t2, -1.0 / 720.0, 1.0 / 24.0), -0.5);
    *cs = fma(e.x, ct, fma(-e.y, st, e.x));
    *sn = fma(e.y, ct, fma(e.x, st, e.y));
}

// 1 / r and, if wanted, r from r^2: one reciprocal square root and a corrected product
// instead of a square root and a division
__device__ __forceinline__ double inv_dist64(double d2) { return rsqrt(d2); }
__device__ __forceinline__ double dist64(double d2, double inv) {
    const double r = d2 * inv;
    // r = 0 where the points coincide (inv is infinite); an integer test, off the FP64 pipe
    return __double_as_longlong(d2) == 0 ? 0.0 : fma(fma(-r, r, d2), 0.5 * inv, r);
}

// w e^{i kappa r} / r (complex) or w / r (real) from r^2
template <bool CPLX>
__device__ __forceinline__ void green64(double d2, double kappa, double w, const double2* __restrict__ tab, double* gr,
                                        double* gi) {
    const double inv = inv_dist64(d2), f = w * inv;
    if constexpr (CPLX) {
        double c, s;
        expi64(kappa * dist64(d2, inv), tab, &c, &s);
        *gr = f * c;
        *gi = f * s;
    } else {
        *gr = f;
        *gi = 0.0;
    }
}

}  // namespace ibem
