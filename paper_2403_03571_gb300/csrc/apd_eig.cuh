// Bounds of the eigenvalues of a symmetric positive-definite 2x2 or 3x3 matrix (FP64 in
// and out).  Host code too, so that the CPU tests run these lines.
#pragma once

#include <math.h>
#include <string.h>

namespace apd {

// The power of two 2^-e that brings a positive finite trace into [1, 2), and 2^e.
// Both products are exact (|e| <= 1000), so a bound of the scaled matrix times 2^e is the
// bound of the matrix itself.
__host__ __device__ __forceinline__ void trace_scale(double trace, double &down, double &up) {
    unsigned long long b;
    memcpy(&b, &trace, sizeof b);
    int e = (int)((b >> 52) & 0x7ffull) - 1023;
    e = e < -1000 ? -1000 : (e > 1000 ? 1000 : e);
    const unsigned long long d = (unsigned long long)(1023 - e) << 52, u = (unsigned long long)(1023 + e) << 52;
    memcpy(&down, &d, sizeof d);
    memcpy(&up, &u, sizeof u);
}

// Lower bound of the smallest eigenvalue, close to it.  2x2: from the characteristic
// quadratic.  3x3, for a trace in [1, 2) (see eigen_bounds): Newton's method on the
// characteristic polynomial f from the left of the smallest root, where f is negative,
// increasing and concave: every iterate stays left of the root, so any number of steps
// gives a lower bound (steps taken 1e-6 short cover their FP32 quotient).  Starts:
// c0 / c1 (between a third of the root and the root; beyond the mean only where rounding
// has eaten c1, and then not taken) and mean - 2 spread.  The FP32 parts want the unit
// scale: det A leaves FP32's range from eigenvalues of 7e12 on, the squared spread below
// 1e-21.
// The FP64 pipe issues a warp instruction every 64 clocks, so the trigonometric
// solution (acos, cos) took 36 us per 1000 seeds against 5 us for this form.
template <int D>
__host__ __device__ __forceinline__ double lambda_min_sym(const double (&s)[D][D]) {
    if (D == 2) {
        const double m = 0.5 * (s[0][0] + s[1][1]);
        const double h = 0.5 * (s[0][0] - s[1][1]);
        const double r = sqrt(h * h + s[0][1] * s[0][1]);
        // m - r computed as det / (m + r) to avoid cancellation
        const double det = s[0][0] * s[1][1] - s[0][1] * s[0][1];
        return (det / (m + r)) * (1.0 - 1e-9);
    } else {
        const double c2 = s[0][0] + s[1][1] + s[2][2];
        const double m01 = s[0][0] * s[1][1] - s[0][1] * s[0][1], m02 = s[0][0] * s[2][2] - s[0][2] * s[0][2],
                     m12 = s[1][1] * s[2][2] - s[1][2] * s[1][2];
        const double c1 = m01 + m02 + m12;
        const double c0 = s[0][0] * m12 - s[0][1] * (s[0][1] * s[2][2] - s[1][2] * s[0][2]) +
                          s[0][2] * (s[0][1] * s[1][2] - s[1][1] * s[0][2]);
        // mean - 2 sqrt(p2 / 6), p2 = ||S - mean I||^2 = ||S||^2 - c2^2 / 3 = 2 (c2^2 / 3 - c1)
        const float q = (float)c2 / 3.f;
        const float p2 = fmaxf((float)(c2 * c2 * (1.0 / 3.0) - c1), 0.f) * (2.f / 6.f);
        const float iso = q - 2.f * sqrtf(p2) - 1e-5f * q;
        const float left = ((float)c0 / (float)c1) * (1.f - 1e-5f);
        const float start = left <= q ? fmaxf(left, iso) : iso;
        double x = fmax((double)start, 0.0);
        float df = 1.f;
#pragma unroll 1
        for (int it = 0; it < 6; ++it) {
            const double f = ((x - c2) * x + c1) * x - c0;
            df = (float)((3.0 * x - 2.0 * c2) * x + c1);
            const float ff = (float)f;
            if (!(df > 0.f) || !(ff < 0.f)) break;
            x += (double)((-ff / df) * (1.f - 1e-6f));
        }
        // the rounding of f near the root: at most 1e-14 c2^3, divided by the slope
        const float c = (float)c2;
        const float slack = 1e-14f * c * c * c / fmaxf(df, 1e-30f);
        return fmax(fmax(x * (1.0 - 1e-9) - (double)slack, (double)iso), 0.0);
    }
}

// Upper bound of the largest eigenvalue: 2x2 m + r; 3x3 (trace in [1, 2)) mean + 2 spread.
template <int D>
__host__ __device__ __forceinline__ double lambda_max_sym(const double (&s)[D][D]) {
    if (D == 2) {
        const double m = 0.5 * (s[0][0] + s[1][1]);
        const double h = 0.5 * (s[0][0] - s[1][1]);
        return (m + sqrt(h * h + s[0][1] * s[0][1])) * (1.0 + 1e-9);
    } else {
        const double p1 = s[0][1] * s[0][1] + s[0][2] * s[0][2] + s[1][2] * s[1][2];
        const double q = (s[0][0] + s[1][1] + s[2][2]) * (1.0 / 3.0);
        const double a0 = s[0][0] - q, a1 = s[1][1] - q, a2 = s[2][2] - q;
        const float p2 = (float)(a0 * a0 + a1 * a1 + a2 * a2 + 2.0 * p1);
        return q * (1.0 + 1e-9) + (double)(2.f * sqrtf(p2 * (1.f / 6.f)) * (1.f + 1e-6f));
    }
}

// lo <= lambda_min(s), hi >= lambda_max(s) at every scale whose determinant FP64 holds; the
// Frobenius norm, which the caller also takes, is another upper bound.
template <int D>
__host__ __device__ __forceinline__ void eigen_bounds(const double (&s)[D][D], double &lo, double &hi) {
    if (D == 2) {
        lo = lambda_min_sym<D>(s);
        hi = lambda_max_sym<D>(s);
    } else {
        double down, up, t[D][D];
        trace_scale(s[0][0] + s[1][1] + s[D - 1][D - 1], down, up);
#pragma unroll
        for (int a = 0; a < D; ++a)
#pragma unroll
            for (int b = 0; b < D; ++b) t[a][b] = s[a][b] * down;
        lo = lambda_min_sym<D>(t) * up;
        hi = lambda_max_sym<D>(t) * up;
    }
}

}  // namespace apd
