// Chebyshev polynomials that precondition the conjugate gradients of the FP64 solves
// (Saad, Iterative Methods for Sparse Linear Systems, algorithm 12.1).
#pragma once

#include <algorithm>
#include <cmath>
#include <utility>
#include <vector>

namespace rve {

// z = M^-1 r: from z_0 = w D^-1 r and d_0 = z_0, for every (c1, c2) of `steps`
//   d <- c1 d + c2 D^-1 (r - A z),  z <- z + d
struct ChebPoly {
    double w = 0.0;
    std::vector<std::pair<float, float>> steps;
};

// The polynomial for the spectrum [lambda / ratio, lambda] of D^-1 A, of degree sqrt(ratio).
//
// lambda is an estimate (a Rayleigh quotient approaches the largest eigenvalue from below),
// so eigenvalues may lie above it.  There the residual polynomial R grows, and 1 - R, the
// eigenvalue of M^-1 A, has the sign of -R: positive for an odd degree, negative for an
// even one.  The degree is odd, so that M stays positive definite whatever the estimate;
// an eigenvalue above it then only stands apart from the others, which costs a few iterations.
// (A plate of 49 665 nodes with one stiff tetrahedron, largest eigenvalue 2.80 against an
// estimate of 2.75, to 1e-10: degree 32 1364 iterations, 322 ms; degree 33 53, 16 ms; Jacobi
// 904, 87 ms.)
inline ChebPoly chebyshev(double lambda, double ratio) {
    ChebPoly p;
    const int degree = std::max(5, (int)std::lround(std::sqrt(ratio))) | 1;
    const double lo = lambda / ratio, th = 0.5 * (lambda + lo), de = 0.5 * (lambda - lo);
    p.w = 1.0 / th;
    double rho = de / th;
    for (int k = 1; k < degree; ++k) {
        const double rn = 1.0 / (2.0 * th / de - rho);
        p.steps.emplace_back((float)(rn * rho), (float)(2.0 * rn / de));
        rho = rn;
    }
    return p;
}

}  // namespace rve
