// sqrt_nodes.h -- nodes and weights of a rational approximation of the square root (host logic, no
// CUDA, so that the tests can compile and check them on the CPU).
//
// Hale, Higham & Trefethen, "Computing A^alpha, log(A), and related matrix functions by contour
// integrals" (SIAM J. Numer. Anal. 2008), method 3: for a symmetric A with spectrum in [m, 1],
//   A^{1/2} ~ sum_j w_j A (A + s_j I)^{-1},   s_j = m (sn/cn)^2(u_j),  w_j = 2 K' sqrt(m) / (pi n) (dn/cn^2)(u_j),
// u_j = (j + 1/2) K' / n, with K' = K(1 - m) and the Jacobi elliptic functions of parameter 1 - m.
// All s_j and w_j are positive; the relative error is about exp(-2 pi^2 n / (6 - ln m)).
#pragma once

#include <cmath>

namespace rpb {

// Spectrum down to 1e-20 of the largest eigenvalue with 128 nodes: error exp(-48), below float64 rounding
// (an eigenvalue under 1e-16 is rounding noise of the matrix anyway).  One node per thread: the four
// warps take the four schedulers of an SM, so fewer nodes would not be faster.
constexpr int kSqrtNodes = 128;
constexpr double kSqrtMin = 1e-20;

struct SqrtNodes {
    double s[kSqrtNodes], w[kSqrtNodes];
};

inline SqrtNodes sqrt_nodes()
{
    const double pi = 3.14159265358979323846, m = kSqrtMin, k1 = std::sqrt(m);
    // K(1 - m) = ln(4/sqrt(m)) + O(m ln m); the elliptic functions from their expansions in the small
    // complementary parameter m (Abramowitz & Stegun 16.15), taken on the lower half of the quarter
    // period, where the neglected m^2 cosh^4(u) is below 1e-18, and reflected to the upper half:
    // (sn/cn)(K' - v) = (cn/sn)(v) / sqrt(m), dn(K' - v) = sqrt(m) / dn(v)
    const double Kp = std::log(4.0 / k1);
    SqrtNodes r;
    for (int j = 0; j < kSqrtNodes / 2; ++j) {
        const double v = (j + 0.5) * Kp / kSqrtNodes;
        const double sh = std::sinh(v), ch = std::cosh(v), q = 0.25 * m * (sh * ch - v);
        const double sc = sh + q * ch;                                     // sn/cn
        const double cn = (1.0 - q * sh / ch) / ch;
        const double dn = (1.0 + 0.25 * m * (sh * ch + v) * sh / ch) / ch;
        const double c = 2.0 * Kp / (pi * kSqrtNodes);
        r.s[j] = m * sc * sc;
        r.w[j] = c * k1 * dn / (cn * cn);
        r.s[kSqrtNodes - 1 - j] = 1.0 / (sc * sc);
        r.w[kSqrtNodes - 1 - j] = c * dn / (sc * sc * cn * cn);
    }
    return r;
}

}  // namespace rpb
