// wide_poly.cuh -- host side of wide_math.cuh's kick integrals: the polynomials behind the
// node sums.  Plain C++.
#pragma once

#include <cmath>
#include <cstring>

namespace fdf {

// g(t) = sum_j W_j (1 + e_j t)^power on [0, 1] as a polynomial of degree kKickDeg: the
// binomial series c_k = binom(power, k) sum_j W_j e_j^k to kSeries terms, whose terms above
// kKickDeg are replaced one by one, from the top, by t^m -> t^m - T*_m(t) 2^(1-2m), T*_m the
// Chebyshev polynomial of [0, 1] (Lanczos' economisation).  Each replacement moves the sum
// by at most |c_m| 2^(1-2m), c_11 the most: below 2^-50 of g for |e_j| <= 0.19.
constexpr int kSeries = 26;

struct ChebStar {
    double c[kSeries + 1][kSeries + 1];     // T*_m(t) 2^(1-2m) = sum_k c[m][k] t^k, c[m][m] = 1
    ChebStar()
    {
        // T*_0 = 1, T*_1 = 2t - 1, T*_{m+1} = 2 (2t - 1) T*_m - T*_{m-1}
        double t0[kSeries + 2] = {1.0}, t1[kSeries + 2] = {-1.0, 2.0};
        std::memset(c, 0, sizeof(c));
        for (int m = 1; m <= kSeries; ++m) {
            for (int k = 0; k <= m; ++k) c[m][k] = std::ldexp(t1[k], 1 - 2 * m);
            double t2[kSeries + 2];
            for (int k = 0; k <= kSeries + 1; ++k) t2[k] = (k ? 4.0 * t1[k - 1] : 0.0) - 2.0 * t1[k] - t0[k];
            std::memcpy(t0, t1, sizeof(t0));
            std::memcpy(t1, t2, sizeof(t1));
        }
    }
};

inline void kick_coef(KickPoly& K, int k, double v)
{
    K.h[k] = (float)v;
    K.l[k] = (float)(v - (double)K.h[k]);
}

// The polynomial times scale; false if |e_j| > 0.19 (its truncation would not stay below 2^-47):
// steps of d ln a above about 0.19 (fewer than 90 from z = 1e9 to 31).
inline bool kick_node_poly(const double* W, const double* e, int n, double power, double scale, KickPoly& K)
{
    static const ChebStar T;
    double c[kSeries + 1], p[8], binom = scale;
    for (int j = 0; j < n; ++j) {
        if (std::fabs(e[j]) > 0.19) return false;
        p[j] = W[j];
    }
    for (int k = 0; k <= kSeries; ++k) {
        double s = 0;
        for (int j = 0; j < n; ++j) {
            s += p[j];
            p[j] *= e[j];
        }
        c[k] = binom * s;
        binom *= (power - k) / (k + 1);
    }
    for (int m = kSeries; m > kKickDeg; --m)
        for (int k = 0; k < m; ++k) c[k] -= c[m] * T.c[m][k];
    for (int k = 0; k <= kKickDeg; ++k) kick_coef(K, k, c[k]);
    return true;
}

}  // namespace fdf
