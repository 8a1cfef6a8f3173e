// One entry of the projection basis in closed form, in fp64 (Section 3.3, Eq. 2-3 with the transforms of Appendix A):
//
//   P[m][n] = (1/N) * [ 1 + 2 * sum_{t=1}^{L-1} cos(pi t (2m+1)/(2L)) * cos(pi t (2n+1)/(2N)) ].
//
// The product of cosines splits into cosines of the sum and difference angle, and each of the
// two cosine series sums to a Dirichlet kernel:
//
//   P[m][n] = (1/(2N)) * [ D(a+) + D(a-) ],   a± = (2m+1) N ± (2n+1) L   (integers),
//   D(a) = sin((2L-1) pi a / (4LN)) / sin(pi a / (4LN)),   D(0) = 2L-1.
//
// 0 < a+ < 4LN and |a-| < 2LN, so the denominator vanishes only at a- = 0.  The numerator's
// phase is reduced exactly in 64-bit integers modulo 8LN before sinpi, so every entry is
// accurate to a few fp64 ulps.
#pragma once

#include <stdint.h>

namespace freqkv {

__device__ inline double dirichlet(int64_t a, int64_t L, int64_t LN4)
{
    if (a < 0) a = -a;  // D is even
    if (a == 0) return (double)(2 * L - 1);
    const int64_t r = ((2 * L - 1) * a) % (2 * LN4);
    return sinpi((double)r / (double)LN4) / sinpi((double)a / (double)LN4);
}

// Retaining components t0 .. t0 + L - 1 instead of the lowest L (the paper's high/low-frequency
// ablation; t0 >= 1 here).  With A = pi (2m+1) / (2L), B = pi (2n+1) / (2N) the orthonormal weights
// give  P[m][n] = (sqrt 2 / N) [ cos(B t0) + sqrt 2 * sum_{t'=1}^{L-1} cos(A t') cos(B (t0 + t')) ],
// and each of the two cosine series the product splits into sums in closed form:
//   sum_{t'=1}^{L-1} cos(theta t' + phi) = sin((L-1) theta / 2) / sin(theta / 2) * cos(L theta / 2 + phi),
// (L - 1) cos(phi) at theta = 0.  All phases are integer multiples of pi / (4LN) and are reduced
// exactly modulo 8LN before sinpi / cospi.
__device__ inline double cos_units(int64_t k, int64_t LN4)
{
    const int64_t period = 2 * LN4;
    k = ((k % period) + period) % period;
    return cospi((double)k / (double)LN4);
}
__device__ inline double sin_units(int64_t k, int64_t LN4)
{
    const int64_t period = 2 * LN4;
    k = ((k % period) + period) % period;
    return sinpi((double)k / (double)LN4);
}
__device__ inline double cosine_series(int64_t a, int64_t phi, int64_t L, int64_t LN4)
{
    if (a == 0) return (double)(L - 1) * cos_units(phi, LN4);
    return sin_units((L - 1) * a, LN4) / sin_units(a, LN4) * cos_units(L * a + phi, LN4);
}

// P[m][n] of the map that keeps components t0 .. t0 + L - 1 of an N-point signal.
__device__ inline double basis_entry(int64_t m, int64_t n, int64_t N, int64_t L, int64_t t0)
{
    const int64_t LN4 = 4 * L * N;
    const int64_t u = (2 * m + 1) * N, w = (2 * n + 1) * L;
    if (t0 == 0) return (dirichlet(u + w, L, LN4) + dirichlet(u - w, L, LN4)) / (double)(2 * N);
    const int64_t phi = (2 * n + 1) * t0 * 2 * L;
    const double series = 0.5 * (cosine_series(u + w, phi, L, LN4) + cosine_series(u - w, -phi, L, LN4));
    return 1.4142135623730951 / (double)N * (cos_units(phi, LN4) + 1.4142135623730951 * series);
}

}  // namespace freqkv
