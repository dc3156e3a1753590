// Free-space mobility of two blobs of the discrete fluid: the 3 x 3 block
// of the blob mobility J L^-1 S that the body-block preconditioner inverts
// (the approach of Kallemov, Bhalla, Griffith and Donev, "An immersed
// boundary method for rigid bodies", 2016: empirical pair functions of the
// grid and kernel in place of the Rotne-Prager-Yamakawa tensor).
//
// M_ij = (f(r) (I - n n^T) + g(r) n n^T) / (eta h), r = |r_i - r_j| / h.
// f and g are the velocity across and along n that a unit force spread by the
// kernel gives a blob at distance r on the MAC grid, averaged over the
// blobs' positions relative to the grid and over directions (periodic box of
// 96 or 128 cells, Hasimoto's correction for its images), at r = 0, 1/4 ..,
// 6; from r = 4 they go over to the Rotne-Prager-Yamakawa tensor, which the
// fluid's response meets to 0.2% there.  Near r = 0 they are flat, where the
// tensor has a corner, so the smallest eigenvalues of M, which set the
// solver's iterations, are up to 20 times smaller than the tensor's: solves
// to 1e-8 of two 42-blob spheres take 20 iterations (27 with the tensor)
// with the three-point kernel and 27 (84) with the six-point kernel.
#pragma once
#include <cmath>

#include "common.cuh"

namespace rbfib {

constexpr int kPairKnots = 25;          // r = 0, 1/4, ..., 6
constexpr double kPairStep = 0.25;

// Cubic pieces of f and g, the blob radius of the tail, and what the
// diagonal of M is raised by (pair_raise).
struct PairMobility {
  double c[2][kPairKnots - 1][4];
  double a, shift;
};

inline void pair_tail(double a, double r, double& f, double& g) {
  f = (1.0 + 2.0 * a * a / (3.0 * r * r)) / (8.0 * M_PI * r);
  g = (1.0 - 2.0 * a * a / (3.0 * r * r)) / (4.0 * M_PI * r);
}

// Cubic spline through the knots, flat at r = 0, with the tail's slope at
// r = 6.
inline PairMobility pair_mobility(int kw) {
  static const double three[2][kPairKnots] = {
    {0.0584973, 0.0572061, 0.0535623, 0.0481889, 0.0420517, 0.0359540, 0.0304755, 0.0259027, 0.0222550,
     0.0194052, 0.0171763, 0.0154186, 0.0139978, 0.0128210, 0.0118300, 0.0109864, 0.0102584, 0.0096237,
     0.0090650, 0.0085699, 0.0081268, 0.0077273, 0.0073650, 0.0070350, 0.0067332},
    {0.0584973, 0.0578241, 0.0559409, 0.0530778, 0.0495507, 0.0456879, 0.0418248, 0.0381751, 0.0348471,
     0.0318880, 0.0292932, 0.0270277, 0.0250510, 0.0233242, 0.0218065, 0.0204639, 0.0192695, 0.0182014,
     0.0172394, 0.0163697, 0.0155805, 0.0148632, 0.0142086, 0.0136095, 0.0130595}};
  static const double six[2][kPairKnots] = {
    {0.0361263, 0.0358104, 0.0348888, 0.0334334, 0.0315512, 0.0293718, 0.0270319, 0.0246577, 0.0223541,
     0.0201998, 0.0182437, 0.0165076, 0.0149924, 0.0136848, 0.0125624, 0.0115992, 0.0107697, 0.0100535,
     0.0094310, 0.0088844, 0.0083996, 0.0079659, 0.0075750, 0.0072204, 0.0068968},
    {0.0361263, 0.0359677, 0.0355013, 0.0347511, 0.0337551, 0.0325604, 0.0312193, 0.0297842, 0.0283041,
     0.0268214, 0.0253708, 0.0239778, 0.0226593, 0.0214250, 0.0202787, 0.0192201, 0.0182456, 0.0173446,
     0.0165107, 0.0157422, 0.0150354, 0.0143857, 0.0137884, 0.0132387, 0.0127322}};
  PairMobility P;
  P.a = kw == 6 ? 1.47 : 0.91;
  P.shift = kw == 6 ? 3e-5 : 2e-4;
  const int n = kPairKnots;
  const double h = kPairStep;
  double lo[2], hi[2];
  pair_tail(P.a, (n - 1) * h - 1e-5, lo[0], lo[1]);
  pair_tail(P.a, (n - 1) * h + 1e-5, hi[0], hi[1]);
  for (int t = 0; t < 2; ++t) {
    const double* y = kw == 6 ? six[t] : three[t];
    const double end = (hi[t] - lo[t]) / 2e-5;
    // second derivatives m: clamped ends, tridiagonal elimination
    double d[kPairKnots], u[kPairKnots], m[kPairKnots];
    d[0] = 0.5;
    u[0] = 3.0 / (h * h) * (y[1] - y[0]);
    for (int i = 1; i < n; ++i) {
      const double rhs = i < n - 1 ? 6.0 / (h * h) * (y[i + 1] - 2.0 * y[i] + y[i - 1])
                                   : 6.0 / h * (end - (y[n - 1] - y[n - 2]) / h);
      const double diag = i < n - 1 ? 4.0 : 2.0;
      d[i] = 1.0 / (diag - d[i - 1]);
      u[i] = (rhs - u[i - 1]) * d[i];
    }
    m[n - 1] = u[n - 1];
    for (int i = n - 2; i >= 0; --i) m[i] = u[i] - d[i] * m[i + 1];
    for (int i = 0; i < n - 1; ++i) {
      double* c = P.c[t][i];
      c[0] = y[i];
      c[1] = (y[i + 1] - y[i]) / h - h / 6.0 * (2.0 * m[i] + m[i + 1]);
      c[2] = 0.5 * m[i];
      c[3] = (m[i + 1] - m[i]) / (6.0 * h);
    }
  }
  return P;
}

__host__ __device__ inline void pair_functions(const PairMobility& P, double r, double& f, double& g) {
  if (r < (kPairKnots - 1) * kPairStep) {
    const int i = (int)(r * (1.0 / kPairStep));
    const double x = r - i * kPairStep;
    const double *cf = P.c[0][i], *cg = P.c[1][i];
    f = fma(fma(fma(cf[3], x, cf[2]), x, cf[1]), x, cf[0]);
    g = fma(fma(fma(cg[3], x, cg[2]), x, cg[1]), x, cg[0]);
  } else {
    const double ir = 1.0 / r, q = P.a * P.a * ir * ir * (2.0 / 3.0), c = ir * (1.0 / (8.0 * M_PI));
    f = c * (1.0 + q);
    g = 2.0 * c * (1.0 - q);
  }
}

// The averages are positive definite only to their statistical error
// (three-point: the grid's own variation), which adds up over blobs that the
// grid does not resolve.  A blob with more than 32 others (itself included)
// within 2 h is raised by that much more: shells of 42 to 800 blobs of radius
// 0.3 to 3 h have smallest eigenvalues down to -7e-4 (500 blobs, radius h / 2)
// before and above zero after it; ordinary shells have about ten.
constexpr double kPairNear = 2.0;
__host__ __device__ inline double pair_raise(const PairMobility& P, int near) {
  return P.shift * (near > 32 ? near / 32.0 : 1.0);
}

// The block of two blobs at d = r_i - r_j (in units of h), in units of
// 1 / (eta h).  Two blobs at one place, whose forces cannot be told apart,
// give NaN: the inversion refuses the matrix.  raise: one blob with itself
// (else 0).
__host__ __device__ inline void pair_block(const PairMobility& P, const double d[3], double raise, double B[9]) {
  const double r2 = d[0] * d[0] + d[1] * d[1] + d[2] * d[2];
  double f, g;
  pair_functions(P, sqrt(r2), f, g);
  const double w = r2 > 0.0 ? (g - f) / r2 : 0.0;
  f = r2 > 0.0 || raise > 0.0 ? f + raise : nan("");
  for (int p = 0; p < 3; ++p)
    for (int q = 0; q < 3; ++q) B[3 * p + q] = (p == q ? f : 0.0) + w * d[p] * d[q];
}

}  // namespace rbfib
