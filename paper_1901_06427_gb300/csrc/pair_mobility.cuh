// Free-space mobility of two blobs of the discrete fluid: the 3 x 3 block
// of the blob mobility J L^-1 S that the body-block preconditioner inverts
// (the approach of Kallemov, Bhalla, Griffith and Donev, "An immersed
// boundary method for rigid bodies", 2016: empirical pair functions of the
// grid and kernel in place of the Rotne-Prager-Yamakawa tensor).
//
// M_ij = (f(r) (I - n n^T) + g(r) n n^T) / (eta h), r = |r_i - r_j| / h.
// f and g are the velocity across and along n that a unit force spread by the
// kernel gives a blob at distance r on the unbounded MAC grid, averaged over
// the blobs' positions relative to the grid and over directions.  With Phi(k)
// the kernel's Fourier transform and K_a = 2 sin(k_a / 2) the average over
// positions is the transform of the positive semidefinite
//   S(k) = Phi(k)^2 (I - K K^T / |K|^2) / |K|^2
// over all of R^3 (the cross terms of different aliases average out), and the
// average over directions keeps only its parts across and along k, both >= 0:
// so every set of distinct blobs has a positive definite M.  Sampled averages
// do not: noise of 1e-6 (six-point) and a tail that sets in over r = 4 .. 6
// made M indefinite for cubes, plates, rods and packed shells.
// Beyond r = 6 f and g are the Rotne-Prager-Yamakawa tensor's of radius P.a.
// Its 1 / r^3 part is larger than the average's, by the dipole tensor times d =
// 0.0562 (six-point), 0.0276 (three-point); so d times the dipole tensor of the
// density (1 - r^2 / 36)^3 (unit integral, r < 6), whose field beyond 6 is
// the point dipole's, is taken off the average: the two meet at 6 without a
// step, at most 0.8% (0.4%) below the average, and only ripples of that
// density's transform at short waves are left below zero (pair_raise).
// A closed shell's uniform normal force, against which the enclosed fluid
// hardly yields, has the smallest mobility, and how small depends on how the
// shell sits on the grid:
// - the three-point table takes half of the average's part along k,
//   compressible motions that the kernel's aliases let through: a shell of 12
//   blobs then has 1.3e-4 (1.9e-4 with all of it; 1.0e-4 on the grid at a sample
//   place); with all of it an ensemble took 2% longer, with none a monolayer 3%;
// - the six-point table adds 1.5e-5 (1 - r/6)^4 (4 r/6 + 1), also positive
//   definite, to f and g: FP32 sweeps stall when M takes a shell of 42 blobs at
//   2e-6 (22 of them refined to 1e-10: 528 iterations without, 192 with; the
//   sampled averages 190).
// Near r = 0 f and g are flat, where the Rotne-Prager-Yamakawa tensor has a
// corner, so the smallest eigenvalues of M, which set the solver's
// iterations, are up to 50 times smaller than the tensor's.  Both constrained
// solves of a step of two 42-blob spheres together: three-point kernel to 1e-8
// 38 iterations, six-point, refined to 1e-10, 104 (with the tensor, and without
// the wall drag in the pressure block, 68 and 404).
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
    {0.058368451, 0.057051804, 0.053397584, 0.048091051, 0.041976915, 0.035878361, 0.030395895, 0.025812222,
     0.022161058, 0.019321777, 0.017112285, 0.015364995, 0.013952638, 0.012786547, 0.011806782, 0.010971495,
     0.010250170, 0.009620144, 0.009064496, 0.008570304, 0.008127448, 0.007727941, 0.007365507, 0.007035210,
     0.006733151},
    {0.058368451, 0.057700866, 0.055811053, 0.052949791, 0.049430216, 0.045591886, 0.041738681, 0.038084725,
     0.034754085, 0.031795648, 0.029204022, 0.026945810, 0.024977833, 0.023256868, 0.021744354, 0.020407704,
     0.019219873, 0.018158529, 0.017205266, 0.016344867, 0.015564695, 0.014854215, 0.014204614, 0.013608474,
     0.013059524}};
  static const double six[2][kPairKnots] = {
    {0.035868804, 0.035554658, 0.034637362, 0.033188571, 0.031316283, 0.029150271, 0.026825876, 0.024469031,
     0.022184819, 0.020050849, 0.018115583, 0.016400845, 0.014907102, 0.013619957, 0.012516480, 0.011570452,
     0.010756071, 0.010050131, 0.009432959, 0.008888509, 0.008404016, 0.007969476, 0.007577136, 0.007221065,
     0.006896825},
    {0.035868804, 0.035711162, 0.035246743, 0.034500010, 0.033508720, 0.032320066, 0.030986148, 0.029559454,
     0.028088919, 0.026616988, 0.025177854, 0.023796872, 0.022490945, 0.021269600, 0.020136448, 0.019090725,
     0.018128725, 0.017244997, 0.016433239, 0.015686939, 0.014999766, 0.014365806, 0.013779673, 0.013236548,
     0.012732174}};
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

// What the diagonal is raised by.  The smallest eigenvalues are those of
// motions that the kernel averages away, next to zero; splines, the step of
// the digits and the changes above move them by less than 1e-5, over cubes of up
// to 11^3 blobs at 0.9 to 1.5 h, plates, slabs, rods, 1200 blobs at random in boxes
// of 6 to 20 h, packed shells: a third of the six-point kernel's shift, a
// twentieth of the other's.  A blob with more than 32 others (itself included)
// within 2 h is raised by that much more: both that and the rounding of the FP32
// inverse grow with the blobs of a cluster (400 at random within h / 5: 2e-5 below
// zero at most, raised by 2.5e-3).
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
