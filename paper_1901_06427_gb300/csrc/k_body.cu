// Coupled body block of the preconditioner for suspensions with few blobs:
// the Schur complement [-M K; K^T 0] of the saddle operator with the blob
// mobility M replaced by the free-space mobility of all blobs of all bodies
// (pair_mobility.cuh; inter-body coupling included).  Built once per
// configuration: dense M; its inverse (FP32) by blocked Gauss-Jordan or, for
// small matrices close to the previous configuration's, by Newton-Schulz
// steps from its inverse; P = M^-1 K; N = (K^T M^-1 K)^-1 (FP64); then one
// matrix that maps the block's input to its output.  Other suspensions use
// one such matrix per body shape.
#include <algorithm>
#include <cmath>
#include <mutex>
#include <utility>

#include <cooperative_groups.h>

#include "common.cuh"
#include "kernels.cuh"
#include "pair_mobility.cuh"

namespace rbfib {

static inline unsigned nblk(i64 n, int bs) { return (unsigned)((n + bs - 1) / bs); }

// M of all blobs, one thread per blob pair.
__global__ void k_mobility_full(int nbl, const double* __restrict__ r, PairMobility P, double ih, double scale,
                                float* __restrict__ M) {
  pdl_entry();
  const i64 t = (i64)blockIdx.x * blockDim.x + threadIdx.x;
  if (t >= (i64)nbl * nbl) return;
  const int i = (int)(t / nbl), j = (int)(t - (i64)i * nbl);
  const double d[3] = {(r[3 * i] - r[3 * j]) * ih, (r[3 * i + 1] - r[3 * j + 1]) * ih, (r[3 * i + 2] - r[3 * j + 2]) * ih};
  double raise = 0.0;
  if (i == j) {
    int near = 0;
    for (int k = 0; k < nbl; ++k) {
      const float x = (float)((r[3 * i] - r[3 * k]) * ih), y = (float)((r[3 * i + 1] - r[3 * k + 1]) * ih),
                  z = (float)((r[3 * i + 2] - r[3 * k + 2]) * ih);
      near += x * x + y * y + z * z < (float)(kPairNear * kPairNear);
    }
    raise = pair_raise(P, near);
  }
  double B[9];
  pair_block(P, d, raise, B);
  float* Mb = M + (i64)(3 * i) * (3 * nbl) + 3 * j;
  for (int p = 0; p < 3; ++p)
    for (int q = 0; q < 3; ++q) Mb[(i64)p * (3 * nbl) + q] = (float)(scale * B[3 * p + q]);
}

// One step of a blocked Gauss-Jordan inversion (no pivoting; the matrices
// are symmetric positive definite, M by its pair functions, with FP32 pivots
// above 4e-5 of the unit of M for 512 blobs in cubes, slabs and dense clusters
// and K^T M^-1 K with it), out of place: with the kGJ pivots from
// k0 (block row and column P), every 32 x 32 tile (I, J) of B is
//   (P, P): D = A_PP^-1;  (P, J): D A_PJ;  (I, P): -A_IP D;
//   (I, J): A_IJ - A_IP D A_PJ.
// Every block inverts the pivot block again (32 pivots, one barrier each,
// two buffers) rather than wait for a launch of its own.  Bound by latency:
// n / 32 launches of a few microseconds, where one block stepping through n
// pivots took 2.35 ms at n = 252 and a chain of FP32 Newton-Schulz products
// (k_ns_gemm) grows with n^3.  Entries past n are those of the identity.
// status = 1 on a zero pivot.
constexpr int kGJ = 32;
template <typename R>
__global__ void __launch_bounds__(256) k_gj_step(int n, int k0, const R* __restrict__ A, R* __restrict__ B,
                                                 int* __restrict__ status) {
  pdl_entry();
  __shared__ R D[2][kGJ][kGJ + 1], U[kGJ][kGJ + 1], L[kGJ][kGJ + 1];
  const int tx = threadIdx.x & 31, ty = threadIdx.x >> 5;
  const int i0 = blockIdx.y * kGJ, j0 = blockIdx.x * kGJ;
  R c[4];
#pragma unroll
  for (int q = 0; q < 4; ++q) {
    const int r = ty + 8 * q;
    const bool rk = k0 + r < n, ri = i0 + r < n, ck = k0 + tx < n, cj = j0 + tx < n;
    D[0][r][tx] = rk && ck ? A[(i64)(k0 + r) * n + k0 + tx] : (r == tx ? R(1) : R(0));
    U[r][tx] = rk && cj ? A[(i64)(k0 + r) * n + j0 + tx] : R(0);
    L[r][tx] = ri && ck ? A[(i64)(i0 + r) * n + k0 + tx] : R(0);
    c[q] = ri && cj ? A[(i64)(i0 + r) * n + j0 + tx] : R(0);
  }
  __syncthreads();
  const int np = min(kGJ, n - k0);
  int cur = 0;
  for (int k = 0; k < np; ++k) {
    const R p = D[cur][k][k];
    const bool ok = p > R(0) || p < R(0);
    if (!ok && threadIdx.x == 0) *status = 1;
    const R ip = ok ? R(1) / p : R(0), row = D[cur][k][tx] * ip;
#pragma unroll
    for (int q = 0; q < 4; ++q) {
      const int r = ty + 8 * q;
      const R f = D[cur][r][k];
      R v;
      if (r == k) v = tx == k ? ip : row;
      else v = tx == k ? -f * ip : D[cur][r][tx] - f * row;
      D[cur ^ 1][r][tx] = v;
    }
    cur ^= 1;
    __syncthreads();
  }
  const bool rowP = i0 == k0, colP = j0 == k0;
  R out[4];
  if (rowP && colP) {
#pragma unroll
    for (int q = 0; q < 4; ++q) out[q] = D[cur][ty + 8 * q][tx];
  } else {
    // left factor D (for the pivot rows) or L, right factor U or D
    R t[4] = {R(0), R(0), R(0), R(0)};
#pragma unroll 8
    for (int k = 0; k < kGJ; ++k) {
      const R u = colP ? D[cur][k][tx] : U[k][tx];
#pragma unroll
      for (int q = 0; q < 4; ++q) t[q] += (colP ? L[ty + 8 * q][k] : D[cur][ty + 8 * q][k]) * u;
    }
    if (rowP) {
#pragma unroll
      for (int q = 0; q < 4; ++q) out[q] = t[q];
    } else if (colP) {
#pragma unroll
      for (int q = 0; q < 4; ++q) out[q] = -t[q];
    } else {
      __syncthreads();
#pragma unroll
      for (int q = 0; q < 4; ++q) U[ty + 8 * q][tx] = t[q];
      __syncthreads();
#pragma unroll 8
      for (int k = 0; k < kGJ; ++k) {
        const R u = U[k][tx];
#pragma unroll
        for (int q = 0; q < 4; ++q) c[q] -= L[ty + 8 * q][k] * u;
      }
#pragma unroll
      for (int q = 0; q < 4; ++q) out[q] = c[q];
    }
  }
#pragma unroll
  for (int q = 0; q < 4; ++q) {
    const int r = i0 + ty + 8 * q;
    if (r < n && j0 + tx < n) B[(i64)r * n + j0 + tx] = out[q];
  }
}

// X = M^-1 (n x n), M kept; tmp: n x n work.
template <typename R>
void gj_inverse(int n, const R* M, R* X, R* tmp, int* status, cudaStream_t s) {
  const int nt = (n + kGJ - 1) / kGJ;
  const R* in = M;
  for (int k = 0; k < nt; ++k) {
    R* out = (nt - 1 - k) % 2 == 0 ? X : tmp;   // the last step lands in X
    launch_k(k_gj_step<R>, dim3(nt, nt), 256, 0, s, n, k * kGJ, in, out, status);
    note_launch();
    in = out;
  }
}

// P = M^-1 K (n3 x 6 nb): column (p, c) of K is nonzero on the blobs of body p
// only: identity for c < 3, w x arm for c >= 3.
__global__ void k_mk(int nbl, int nb, const int* __restrict__ boff, const double* __restrict__ arm,
                     const float* __restrict__ Mi, float* __restrict__ P) {
  pdl_entry();
  const i64 n3 = 3 * (i64)nbl, m = 6 * (i64)nb;
  const i64 t = (i64)blockIdx.x * blockDim.x + threadIdx.x;
  if (t >= n3 * m) return;
  const int row = (int)(t / m), col = (int)(t - (i64)row * m);
  const int p = col / 6, c = col % 6;
  double acc = 0.0;
  for (int i = boff[p]; i < boff[p + 1]; ++i) {
    const float* Mr = Mi + (i64)row * n3 + 3 * i;
    if (c < 3) {
      acc += Mr[c];
    } else {
      // (w x arm) for w = e_{c-3}: e_x x d = (0, -dz, dy), e_y x d = (dz, 0, -dx), e_z x d = (-dy, dx, 0)
      const double* d = arm + 3 * i;
      double k0, k1, k2;
      if (c == 3) { k0 = 0; k1 = -d[2]; k2 = d[1]; }
      else if (c == 4) { k0 = d[2]; k1 = 0; k2 = -d[0]; }
      else { k0 = -d[1]; k1 = d[0]; k2 = 0; }
      acc += Mr[0] * k0 + Mr[1] * k1 + Mr[2] * k2;
    }
  }
  P[t] = (float)acc;
}

// A = K^T P (6 nb x 6 nb, FP64)
__global__ void k_ktp(int nbl, int nb, const int* __restrict__ boff, const double* __restrict__ arm,
                      const float* __restrict__ P, double* __restrict__ A) {
  pdl_entry();
  const int m = 6 * nb;
  const int t = blockIdx.x * blockDim.x + threadIdx.x;
  if (t >= m * m) return;
  const int row = t / m, col = t - row * m;
  const int p = row / 6, c = row % 6;
  double acc = 0.0;
  for (int i = boff[p]; i < boff[p + 1]; ++i) {
    const double x = P[(i64)(3 * i) * m + col], y = P[(i64)(3 * i + 1) * m + col], z = P[(i64)(3 * i + 2) * m + col];
    const double* d = arm + 3 * i;
    if (c == 0) acc += x;
    else if (c == 1) acc += y;
    else if (c == 2) acc += z;
    else if (c == 3) acc += d[1] * z - d[2] * y;
    else if (c == 4) acc += d[2] * x - d[0] * z;
    else acc += d[0] * y - d[1] * x;
  }
  A[t] = acc;
}

// Square FP32 products for the Newton-Schulz update of the inverse
// (n x n, row-major): MODE 0 forms C = I - A B and adds sum(C_ij^2) to
// *ss; MODE 1 forms C = D + A B.  16 x 16 output tiles on 64 threads (a
// 2 x 2 block of outputs each), so that even n = 252 spreads over 256 CTAs;
// the A rows and B columns of a tile are staged through shared memory in
// k-slices of up to kNSK (one slice for n <= kNSK, all of its loads in
// flight at once), A transposed so that a thread reads its two rows and its
// two columns of a k step as two 8-byte loads.  Entries past n are
// zero-filled.  n <= 1536: these products take microseconds, so they stay
// on the FP32 pipe.
constexpr int kNSTile = 16, kNSK = 256, kNSPad = kNSTile + 2;
template <int MODE>
__global__ void __launch_bounds__(64) k_ns_gemm(int n, const float* __restrict__ A, const float* __restrict__ B,
                                                const float* __restrict__ D, float* __restrict__ C,
                                                double* __restrict__ ss) {
  pdl_entry();
  __shared__ __align__(16) float As[kNSK][kNSPad];   // As[k][r] = A[r0 + r][k0 + k]
  __shared__ __align__(16) float Bs[kNSK][kNSTile];  // Bs[k][c] = B[k0 + k][c0 + c]
  __shared__ double red[2];
  const int tid = threadIdx.x, tx = tid & 7, ty = tid >> 3;
  const int r0 = blockIdx.y * kNSTile, c0 = blockIdx.x * kNSTile;
  float acc[2][2] = {{0.f, 0.f}, {0.f, 0.f}};
  for (int k0 = 0; k0 < n; k0 += kNSK) {
    const int kc = min(kNSK, n - k0);
    // Thread tid stages elements tid + 64 q (q < 64) of each slice, in two
    // batches of 32 loads per matrix held in registers, so that the loads
    // of a batch are in flight together.  A: consecutive threads along k
    // (element (r, kk) = (q / 4, 64 (q % 4) + tid), coalesced rows of A);
    // B: consecutive threads along the tile's columns ((kk, c) =
    // (4 q + tid / 16, tid % 16)).
#pragma unroll
    for (int h = 0; h < 2; ++h) {
      float ra[32], rb[32];
#pragma unroll
      for (int q = 0; q < 32; ++q) {
        const int qq = 32 * h + q;
        const int r = qq >> 2, ka = 64 * (qq & 3) + tid;
        const int kb = 4 * qq + (tid >> 4), c = tid & 15;
        ra[q] = (ka < kc && r0 + r < n) ? A[(i64)(r0 + r) * n + k0 + ka] : 0.f;
        rb[q] = (kb < kc && c0 + c < n) ? B[(i64)(k0 + kb) * n + c0 + c] : 0.f;
      }
#pragma unroll
      for (int q = 0; q < 32; ++q) {
        const int qq = 32 * h + q;
        As[64 * (qq & 3) + tid][qq >> 2] = ra[q];
        Bs[4 * qq + (tid >> 4)][tid & 15] = rb[q];
      }
    }
    __syncthreads();
#pragma unroll 8
    for (int kk = 0; kk < kc; ++kk) {
      const float2 a = *reinterpret_cast<const float2*>(&As[kk][2 * ty]);
      const float2 b = *reinterpret_cast<const float2*>(&Bs[kk][2 * tx]);
      acc[0][0] = fmaf(a.x, b.x, acc[0][0]);
      acc[0][1] = fmaf(a.x, b.y, acc[0][1]);
      acc[1][0] = fmaf(a.y, b.x, acc[1][0]);
      acc[1][1] = fmaf(a.y, b.y, acc[1][1]);
    }
    __syncthreads();
  }
  double sq = 0.0;
#pragma unroll
  for (int u = 0; u < 2; ++u)
#pragma unroll
    for (int q = 0; q < 2; ++q) {
      const int row = r0 + 2 * ty + u, col = c0 + 2 * tx + q;
      if (row >= n || col >= n) continue;
      const i64 o = (i64)row * n + col;
      float v;
      if (MODE == 0) {
        v = (row == col ? 1.f : 0.f) - acc[u][q];
        sq += (double)v * (double)v;
      } else {
        v = D[o] + acc[u][q];
      }
      C[o] = v;
    }
  if (MODE == 0) {
    for (int o = 16; o > 0; o >>= 1) sq += __shfl_xor_sync(0xffffffffu, sq, o);
    if ((tid & 31) == 0) red[tid >> 5] = sq;
    __syncthreads();
    if (tid == 0) atomicAdd(ss, red[0] + red[1]);
  }
}

template <int MODE>
void ns_gemm(int n, const float* A, const float* B, const float* D, float* C, double* ss, cudaStream_t s) {
  const unsigned nt = (unsigned)((n + kNSTile - 1) / kNSTile);
  launch_k(k_ns_gemm<MODE>, dim3(nt, nt), 64, 0, s, n, A, B, D, C, ss);
  note_launch();
}

// Rotates the previous configuration's inverse with each body's rotation
// since then: X_ij <- D_b(i) X_ij D_b(j)^T for the 3 x 3 blocks (blobs i, j
// of bodies b(i), b(j)), D_p = R(quat_new_p) R(quat_old_p)^T.  M's blocks
// are rotation-covariant, so rotating each body rigidly about its centre turns
// the intra-body blocks of M into exactly these; for a single body the
// rotated inverse is exact.  With several bodies the start's error comes from
// the inter-body blocks of M, which the move also changes.  One thread per
// block, in place.
__global__ void k_rotate_inverse(int nbl, const int* __restrict__ bob, const double* __restrict__ qnew,
                                 const double* __restrict__ qold, float* __restrict__ X) {
  pdl_entry();
  const i64 t = (i64)blockIdx.x * blockDim.x + threadIdx.x;
  if (t >= (i64)nbl * nbl) return;
  const int i = (int)(t / nbl), j = (int)(t - (i64)i * nbl);
  double D[2][9];
  const int body[2] = {bob[i], bob[j]};
  for (int s = 0; s < 2; ++s) {
    double Rn[9], Ro[9];
    quat_rot(qnew + 4 * body[s], Rn);
    quat_rot(qold + 4 * body[s], Ro);
    for (int a = 0; a < 3; ++a)
      for (int b = 0; b < 3; ++b)
        D[s][3 * a + b] = Rn[3 * a] * Ro[3 * b] + Rn[3 * a + 1] * Ro[3 * b + 1] + Rn[3 * a + 2] * Ro[3 * b + 2];
  }
  const i64 n3 = 3 * (i64)nbl;
  float* Xb = X + (3 * (i64)i) * n3 + 3 * (i64)j;
  double x[9], y[9];
  for (int a = 0; a < 3; ++a)
    for (int b = 0; b < 3; ++b) x[3 * a + b] = (double)Xb[a * n3 + b];
  // y = D_i x D_j^T
  for (int a = 0; a < 3; ++a)
    for (int b = 0; b < 3; ++b) {
      double acc = 0.0;
      for (int c = 0; c < 3; ++c)
        for (int e = 0; e < 3; ++e) acc += D[0][3 * a + c] * x[3 * c + e] * D[1][3 * b + e];
      y[3 * a + b] = acc;
    }
  for (int a = 0; a < 3; ++a)
    for (int b = 0; b < 3; ++b) Xb[a * n3 + b] = (float)y[3 * a + b];
}

// Build the coupled body block for a new configuration: M^-1, P = M^-1 K and
// N = (K^T M^-1 K)^-1.
//  - warm (small matrices, dense_body_warm): Minv holds the inverse of the
//    previous configuration's M, built at the body orientations qold (NULL:
//    unknown).  The start X0 is that inverse rotated with each body's
//    rotation since (k_rotate_inverse).  If ||R0||_F = ||I - M X0||_F (which
//    bounds the spectral norm) is at most kNSMaxStart, kNSIters Newton-Schulz
//    steps X <- X + X (I - M X) leave at most kNSMaxStart^(2^kNSIters) (FP32
//    roundoff in practice).
//  - otherwise, or when R0 is larger (a first configuration, a large move):
//    blocked Gauss-Jordan (k_gj_step).
// Mw, Tw, Uw: n3 x n3 FP32 work matrices; Nw: 2 (6 nb)^2 FP64; ss: one device
// double; ss_host: pinned host double (the choice needs one read of ||R0||).
constexpr double kNSMaxStart = 0.25;
constexpr int kNSIters = 4;   // even: the result lands in Minv
// Up to this size the warm start's eight products take about as long as the
// blocked inversion (40 us each at n = 252); above it they grow with n^3
// while the inversion's launches grow with n.
// With this M the start is close after small moves only: two 42-blob spheres'
// Brownian steps (0.05 h, 0.016 rad) leave ||R0||_F at 2 to 4 and are inverted
// anew, a hundredth of them 0.02 to 0.04.
constexpr int kNSMaxRows = 256;
bool dense_body_warm(int nbl) { return 3 * nbl <= kNSMaxRows; }
// The pieces of the set-up, also used one by one by the device-driven SEM
// step (where the warm-start decision is an IF/ELSE graph node).
void dense_body_mobility(int nbl, const double* r, const PairMobility& pm, double h, double eta, float* Mw,
                         cudaStream_t s) {
  launch_k(k_mobility_full, nblk((i64)nbl * nbl, 128), 128, 0, s, nbl, r, pm, 1.0 / h, 1.0 / (eta * h), Mw);
  note_launch();
}
// Warm start: X0 = Minv rotated with each body's rotation since it was built
// (when qnew and qold are known), and Tw = R0 = I - M X0 with ss[0] = ||R0||_F^2.
void dense_body_warm_start(int nbl, const int* bob, const double* qnew, const double* qold, float* Minv,
                           const float* Mw, float* Tw, double* ss, cudaStream_t s) {
  if (qnew && qold) {
    launch_k(k_rotate_inverse, nblk((i64)nbl * nbl, 128), 128, 0, s, nbl, bob, qnew, qold, Minv);
    note_launch();
  }
  cudaMemsetAsync(ss, 0, sizeof(double), s);
  ns_gemm<0>(3 * nbl, Mw, Minv, nullptr, Tw, ss, s);
}
// kNSIters Newton-Schulz steps from X0 = Minv with R0 in Tw; the result
// lands in Minv (kNSIters is even).
void dense_body_ns(int nbl, float* Minv, const float* Mw, float* Tw, float* Uw, double* ss, cudaStream_t s) {
  const int n3 = 3 * nbl;
  float* X = Minv;
  float* Y = Uw;
  for (int it = 0; it < kNSIters; ++it) {
    if (it > 0) ns_gemm<0>(n3, Mw, X, nullptr, Tw, ss, s);   // R = I - M X
    ns_gemm<1>(n3, X, Tw, X, Y, nullptr, s);                 // X' = X + X R
    float* t = X; X = Y; Y = t;
  }
}
void dense_body_gj(int nbl, float* Minv, const float* Mw, float* Uw, int* status, cudaStream_t s) {
  gj_inverse<float>(3 * nbl, Mw, Minv, Uw, status, s);
}
// P = M^-1 K and N = (K^T P)^-1 (FP64; status = 1 on a zero pivot).
void dense_body_finish(int nbl, int nb, const int* boff, const double* arm, const float* Minv, float* P, double* N,
                       double* Nw, int* status, cudaStream_t s) {
  const i64 n3 = 3 * (i64)nbl, m = 6 * (i64)nb;
  launch_k(k_mk, nblk(n3 * m, 256), 256, 0, s, nbl, nb, boff, arm, Minv, P);
  note_launch();
  launch_k(k_ktp, nblk(m * m, 256), 256, 0, s, nbl, nb, boff, arm, P, Nw);
  note_launch();
  gj_inverse<double>((int)m, Nw, N, Nw + m * m, status, s);
}

// IF/ELSE condition of the device-driven warm start: ||R0||_F <= kNSMaxStart;
// warm[0] counts the builds that take the Newton-Schulz branch.
__global__ void k_ns_decide(const double* ss, cudaGraphConditionalHandle h, long long* warm) {
  pdl_entry();
  if (threadIdx.x != 0 || blockIdx.x != 0) return;
  const bool ok = ss[0] <= kNSMaxStart * kNSMaxStart;
  if (ok) warm[0] += 1;
  cudaGraphSetConditional(h, ok ? 1u : 0u);
}
void ns_decide(const double* ss, cudaGraphConditionalHandle h, long long* warm, cudaStream_t s) {
  launch_k(k_ns_decide, 1, 32, 0, s, ss, h, warm);
  note_launch();
}

cudaError_t dense_body_build(int nbl, int nb, const int* boff, const int* bob, const double* r, const double* arm,
                             const double* qnew, const double* qold, const PairMobility& pm, double h, double eta,
                             float* Minv, float* P, double* N, int* status, float* Mw, float* Tw, float* Uw,
                             double* Nw, double* ss, double* ss_host, bool warm, cudaStream_t s, bool* used_out) {
  cudaError_t e;
#define RB_CK(call)                      \
  if ((e = (call)) != cudaSuccess) return e
  RB_CK(cudaMemsetAsync(status, 0, sizeof(int), s));
  bool used = false;
  *used_out = false;
  dense_body_mobility(nbl, r, pm, h, eta, Mw, s);
  if (warm && dense_body_warm(nbl)) {
    dense_body_warm_start(nbl, bob, qnew, qold, Minv, Mw, Tw, ss, s);
    RB_CK(cudaMemcpyAsync(ss_host, ss, sizeof(double), cudaMemcpyDeviceToHost, s));
    RB_CK(cudaStreamSynchronize(s));
    used = std::sqrt(std::max(ss_host[0], 0.0)) <= kNSMaxStart;
  }
  if (used) dense_body_ns(nbl, Minv, Mw, Tw, Uw, ss, s);
  else dense_body_gj(nbl, Minv, Mw, Uw, status, s);
  dense_body_finish(nbl, nb, boff, arm, Minv, P, N, Nw, status, s);
  *used_out = used;
  return cudaGetLastError();
#undef RB_CK
}

// The block as one matrix.  With P = M^-1 K and N = (K^T P)^-1 the solution
// of [-M K; K^T 0] (lambda, U) = (-s, r_U) is linear in (s, r_U):
//   [lambda]   [E P^T - M^-1  E] [s  ]
//   [U     ] = [E^T           N] [r_U],   E = P N,
// so one product replaces the chain M^-1 s -> K^T -> N -> P U - t, whose four
// dependent steps cost a cluster barrier or a run of FP64 latency each.
// The rows of lambda are FP32 (B), as the chain's products with M^-1 and P
// were; the rows of U, (E^T N), are held and summed in FP64 (G), as the chain's
// K^T, N and U were.
// E: one thread per entry, FP64 sums; its transpose goes to G, rows of ldg.
__global__ void k_body_e(int n3, int m, int ldg, const float* __restrict__ P, const double* __restrict__ N,
                         float* __restrict__ E, double* __restrict__ G) {
  pdl_entry();
  const i64 t = (i64)blockIdx.x * blockDim.x + threadIdx.x;
  if (t >= (i64)n3 * m) return;
  const int r = (int)(t / m), c = (int)(t - (i64)r * m);
  double a0 = 0.0, a1 = 0.0;
  int k = 0;
  for (; k + 1 < m; k += 2) {
    a0 = fma((double)P[(i64)r * m + k], N[(i64)k * m + c], a0);
    a1 = fma((double)P[(i64)r * m + k + 1], N[(i64)(k + 1) * m + c], a1);
  }
  if (k < m) a0 = fma((double)P[(i64)r * m + k], N[(i64)k * m + c], a0);
  E[t] = (float)(a0 + a1);
  G[(i64)c * ldg + r] = a0 + a1;
  if (r < m) G[(i64)c * ldg + n3 + r] = N[(i64)c * m + r];   // m <= n3: three blobs a body at least
}

// The rows of lambda, B (n3 rows of ld floats), 32 x 32 tiles of 256 threads.
__global__ void __launch_bounds__(256) k_body_matrix(int n3, int m, int ld, const float* __restrict__ Mi,
                                                     const float* __restrict__ P, const float* __restrict__ E,
                                                     float* __restrict__ B) {
  pdl_entry();
  __shared__ float Es[32][33], Ps[32][33];
  const int tx = threadIdx.x & 31, ty = threadIdx.x >> 5;
  const int r0 = blockIdx.y * 32, c0 = blockIdx.x * 32, n = n3 + m;
  float acc[4] = {0.f, 0.f, 0.f, 0.f};
  for (int k0 = 0; k0 < m; k0 += 32) {
#pragma unroll
    for (int q = 0; q < 4; ++q) {
      const int r = r0 + ty + 8 * q, c = c0 + ty + 8 * q, k = k0 + tx;
      Es[ty + 8 * q][tx] = r < n3 && k < m ? E[(i64)r * m + k] : 0.f;
      Ps[ty + 8 * q][tx] = c < n3 && k < m ? P[(i64)c * m + k] : 0.f;
    }
    __syncthreads();
    for (int k = 0; k < 32; ++k)
#pragma unroll
      for (int q = 0; q < 4; ++q) acc[q] = fmaf(Es[ty + 8 * q][k], Ps[tx][k], acc[q]);
    __syncthreads();
  }
  const int c = c0 + tx;
#pragma unroll
  for (int q = 0; q < 4; ++q) {
    const int r = r0 + ty + 8 * q;
    if (r >= n3 || c >= ld) continue;
    float v = 0.f;
    if (c < n) v = c < n3 ? acc[q] - Mi[(i64)r * n3 + c] : E[(i64)r * m + c - n3];
    B[(i64)r * ld + c] = v;
  }
}

void dense_body_matrix(int nbl, int nb, const float* Minv, const float* P, const double* N, float* E, float* B,
                       double* G, cudaStream_t s) {
  const int n3 = 3 * nbl, m = 6 * nb, ld = body_ld(n3 + m);
  launch_k(k_body_e, nblk((i64)n3 * m, 256), 256, 0, s, n3, m, ld, P, N, E, G);
  note_launch();
  launch_k(k_body_matrix, dim3((ld + 31) / 32, (n3 + 31) / 32), 256, 0, s, n3, m, ld, Minv, P, E, B);
  note_launch();
}

// One row of the block's matrix times x (shared memory), by a warp; the row's
// first kBodyPre 16-byte words of each lane come from registers.
constexpr int kBodyPre = 3;
RBFIB_DEVFN float4 body_word(const float* __restrict__ row, int ld, int w) {
  return 4 * w < ld ? __ldg(reinterpret_cast<const float4*>(row) + w) : make_float4(0.f, 0.f, 0.f, 0.f);
}
RBFIB_DEVFN float body_row(const float* __restrict__ row, const float4 pre[kBodyPre], const float* x, int ld, int lane) {
  float a[4] = {0.f, 0.f, 0.f, 0.f};
  auto add = [&](const float4& b, int w) {
    if (4 * w >= ld) return;
    const float4 v = *reinterpret_cast<const float4*>(x + 4 * w);
    a[0] = fmaf(b.x, v.x, a[0]);
    a[1] = fmaf(b.y, v.y, a[1]);
    a[2] = fmaf(b.z, v.z, a[2]);
    a[3] = fmaf(b.w, v.w, a[3]);
  };
#pragma unroll
  for (int q = 0; q < kBodyPre; ++q) add(pre[q], lane + 32 * q);
  for (int w = lane + 32 * kBodyPre; 4 * w < ld; w += 32) add(body_word(row, ld, w), w);
  float t = (a[0] + a[1]) + (a[2] + a[3]);
#pragma unroll
  for (int o = 16; o > 0; o >>= 1) t += __shfl_xor_sync(0xffffffffu, t, o);
  return t;
}

// One row of G (n doubles) times x (shared memory) by L lanes, lane l of them;
// a lane's first kBodyPre64 entries come from registers, the others in batches
// whose loads are in flight together.  Every lane gets the product.
constexpr int kBodyPre64 = 4;
template <int L>
RBFIB_DEVFN void body_words64(const double* __restrict__ g, int c, int n, double w[kBodyPre64]) {
#pragma unroll
  for (int u = 0; u < kBodyPre64; ++u) w[u] = c + L * u < n ? __ldg(g + c + L * u) : 0.0;
}
template <int L, typename X>
RBFIB_DEVFN double body_row64(const double* __restrict__ g, double w[kBodyPre64], const X* x, int n, int l) {
  double a[kBodyPre64] = {0.0, 0.0, 0.0, 0.0};
  for (int c = l; c < n; c += L * kBodyPre64) {
    if (c != l) body_words64<L>(g, c, n, w);
#pragma unroll
    for (int u = 0; u < kBodyPre64; ++u)
      if (c + L * u < n) a[u] = fma(w[u], (double)x[c + L * u], a[u]);
  }
  double t = (a[0] + a[1]) + (a[2] + a[3]);
#pragma unroll
  for (int o = L / 2; o > 0; o >>= 1) t += __shfl_xor_sync(0xffffffffu, t, o);
  return t;
}

// Coupled block, z = (B; G) (r_lambda + J v, r_U).  Every cluster of 8 CTAs forms
// the whole input, one warp per blob component over the cluster, each value
// written to all eight CTAs through distributed shared memory; after the one
// cluster barrier (the gather's latency hides the first rows' loads, issued
// before it) the rows of B and G are split over the CTAs of all clusters.
constexpr int kBodyCtas = 8, kBodyThreads = 512;
__global__ void __cluster_dims__(kBodyCtas, 1, 1) __launch_bounds__(kBodyThreads)
    k_dense_body_apply(int n3, int m, int ld, const float* __restrict__ B, const double* __restrict__ G,
                       const float* __restrict__ r, float* __restrict__ z, double* __restrict__ z64, Dims d,
                       const BlobStencil<float>* __restrict__ tab, const float* __restrict__ v) {
  pdl_entry();
  namespace cg = cooperative_groups;
  cg::cluster_group cl = cg::this_cluster();
  extern __shared__ __align__(16) double svd[];   // the input in FP64 (ld), then in FP32
  float* sv = reinterpret_cast<float*>(svd + ld);
  const int n = n3 + m;
  const int rpc = (n3 + gridDim.x - 1) / gridDim.x;
  const int r0 = blockIdx.x * rpc, r1 = min(n3, r0 + rpc);
  const int lane = threadIdx.x & 31, wid = threadIdx.x >> 5, nw = kBodyThreads / 32;
  // every CTA of the cluster must have started before its memory is written
  auto started = cl.barrier_arrive();
  float4 pre[kBodyPre];
  // the last nu warps take the CTA's share of the rows of G, the others that of B
  const int nu = min(nw / 2, (m + (int)gridDim.x - 1) / (int)gridDim.x), nr = nw - nu;
  if (wid < nr && r0 + wid < r1)
#pragma unroll
    for (int q = 0; q < kBodyPre; ++q) pre[q] = body_word(B + (i64)(r0 + wid) * ld, ld, lane + 32 * q);
  const int u0 = wid < nr ? m : (int)blockIdx.x + (int)gridDim.x * (wid - nr);
  double gw[kBodyPre64];
  if (u0 < m) body_words64<32>(G + (i64)u0 * ld, lane, n, gw);
  cl.barrier_wait(std::move(started));
  for (int c = (int)cl.block_rank() * nw + wid; c < n3; c += kBodyCtas * nw) {
    const float s = r[c] + warp_interp<float>(d, c % 3, tab + c, v, lane);
    if (lane < kBodyCtas) {
      cl.map_shared_rank(sv, lane)[c] = s;
      cl.map_shared_rank(svd, lane)[c] = (double)s;
    }
  }
  for (int i = n3 + threadIdx.x; i < ld; i += kBodyThreads) {
    sv[i] = i < n ? r[i] : 0.f;
    svd[i] = (double)sv[i];
  }
  cl.sync();
  for (int u = u0; u < m; u += (int)gridDim.x * nu) {
    if (u != u0) body_words64<32>(G + (i64)u * ld, lane, n, gw);
    const double t = body_row64<32>(G + (i64)u * ld, gw, svd, n, lane);
    if (lane == 0) {
      z[n3 + u] = (float)t;
      if (z64) z64[n3 + u] = (double)(float)t;
    }
  }
  for (int row = wid < nr ? r0 + wid : r1; row < r1; row += nr) {
    if (row != r0 + wid)
#pragma unroll
      for (int q = 0; q < kBodyPre; ++q) pre[q] = body_word(B + (i64)row * ld, ld, lane + 32 * q);
    const float t = body_row(B + (i64)row * ld, pre, sv, ld, lane);
    if (lane == 0) {
      z[row] = t;
      if (z64) z64[row] = (double)t;
    }
  }
}

void dense_body_apply(int nbl, int nb, const float* B, const double* G, const float* r, float* z, double* z64,
                      const Dims& d, const BlobStencil<float>* tab, const float* v, cudaStream_t s) {
  const int n3 = 3 * nbl, m = 6 * nb, ld = body_ld(n3 + m);
  // about four rows of B per warp and 4096 FP64 products (1 us of the pipe)
  // per CTA at most
  const int rows = 4 * kBodyCtas * (kBodyThreads / 32), products = 4096 * kBodyCtas;
  const int clusters = std::min(152 / kBodyCtas, std::max((n3 + rows - 1) / rows, (m * (n3 + m) + products - 1) / products));
  launch_k(k_dense_body_apply, kBodyCtas * clusters, kBodyThreads, (sizeof(double) + sizeof(float)) * ld, s, n3, m, ld, B, G,
           r, z, z64, d, tab, v);
  note_launch();
}

// Per-body block: the matrices of each body's shape in the body frame (B_s of
// 3 blobs rows, G_s of 6; host-built, all shapes one after the other), one
// CTA per body: input gathered, its three-vectors (blob velocities, force,
// torque) turned into the body frame, product, turned back.
__global__ void __launch_bounds__(512) k_body_apply(int nbl, const int* __restrict__ boff, const int* __restrict__ shape_of,
                                                    const i64* __restrict__ shape_off, const float* __restrict__ Bs,
                                                    const i64* __restrict__ shape_offg, const double* __restrict__ Gs,
                                                    const double* __restrict__ quat, const float* __restrict__ r,
                                                    float* __restrict__ z, double* __restrict__ z64, Dims d,
                                                    const BlobStencil<float>* __restrict__ tab, const float* __restrict__ vel) {
  pdl_entry();
  extern __shared__ __align__(16) float sh[];
  const int p = blockIdx.x, b0 = boff[p], n3 = 3 * (boff[p + 1] - b0), n = n3 + 6, ld = body_ld(n);
  const float* B = Bs + shape_off[shape_of[p]];
  const double* G = Gs + shape_offg[shape_of[p]];
  float* x = sh;            // input in the lab, later lambda in the body frame
  float* y = sh + ld;       // input in the body frame
  __shared__ double U[8];   // U in the body frame
  const int lane = threadIdx.x & 31, wid = threadIdx.x >> 5, nw = blockDim.x >> 5;
  float4 pre[kBodyPre];
  if (wid < min(n3, nw - 2))
#pragma unroll
    for (int q = 0; q < kBodyPre; ++q) pre[q] = body_word(B + (i64)wid * ld, ld, lane + 32 * q);
  // rows of U, eight lanes each (few lanes of the two-lane FP64 pipe go to the
  // sums over lanes): four by the last warp, two by the one before, which take
  // no rows of B (with some of them one sphere's solve in a 32^3 box took 2.72 ms,
  // now 2.68)
  const int u = min(4 * (nw - 1 - wid) + (lane >> 3), 5);
  double gw[kBodyPre64];
  if (wid >= nw - 2) body_words64<8>(G + (i64)u * ld, lane & 7, n, gw);
  // FP64 costs a warp instruction whatever its lanes do: the rotation by one
  // warp, the turns by one thread per component
  __shared__ double R[9];
  if (wid == nw - 1) {
    double Rr[9];
    quat_rot(quat + 4 * p, Rr);
#pragma unroll
    for (int i = 0; i < 9; ++i)
      if (lane == i) R[i] = Rr[i];
  }
  for (int c = wid; c < n3; c += nw) {
    const float s = r[3 * b0 + c] + warp_interp<float>(d, c % 3, tab + 3 * b0 + c, vel, lane);
    if (lane == 0) x[c] = s;
  }
  if (threadIdx.x < 6) x[n3 + threadIdx.x] = r[3 * nbl + 6 * p + threadIdx.x];
  if (n + (int)threadIdx.x < ld) y[n + threadIdx.x] = 0.f;
  __syncthreads();
  for (int t = threadIdx.x; t < n; t += blockDim.x) {
    const int i = t / 3, a = t - 3 * i;
    y[t] = (float)(R[a] * (double)x[3 * i] + R[3 + a] * (double)x[3 * i + 1] + R[6 + a] * (double)x[3 * i + 2]);
  }
  __syncthreads();
  if (wid >= nw - 2) {
    const double t = body_row64<8>(G + (i64)u * ld, gw, y, n, lane & 7);
    if ((lane & 7) == 0) U[4 * (nw - 1 - wid) + (lane >> 3)] = t;
  }
  for (int row = wid < nw - 2 ? wid : n3; row < n3; row += nw - 2) {
    if (row != wid)
#pragma unroll
      for (int q = 0; q < kBodyPre; ++q) pre[q] = body_word(B + (i64)row * ld, ld, lane + 32 * q);
    const float t = body_row(B + (i64)row * ld, pre, y, ld, lane);
    if (lane == 0) x[row] = t;
  }
  __syncthreads();
  for (int t = threadIdx.x; t < n; t += blockDim.x) {
    const int i = t / 3, a = t - 3 * i;
    double w[3];
#pragma unroll
    for (int c = 0; c < 3; ++c) w[c] = t < n3 ? (double)x[3 * i + c] : U[3 * i + c - n3];
    const float v = (float)(R[3 * a] * w[0] + R[3 * a + 1] * w[1] + R[3 * a + 2] * w[2]);
    const i64 o = t < n3 ? 3 * (i64)b0 + t : 3 * (i64)nbl + 6 * p + t - n3;
    z[o] = v;
    if (z64) z64[o] = (double)v;
  }
}

void body_apply(const BodyView& b, const ShapeView& sv, const float* r, float* z, double* z64, const Dims& d,
                const float* v, cudaStream_t s) {
  const size_t shm = 2 * sizeof(float) * (size_t)body_ld(3 * sv.max_blobs + 6);
  static std::once_flag f;
  std::call_once(f, [] { cudaFuncSetAttribute(k_body_apply, cudaFuncAttributeMaxDynamicSharedMemorySize, kBodyMaxSmem); });
  // a body's gathers and rows are dealt to its warps one after another, so
  // larger bodies take more of them (one 42-blob sphere's mobility solve in a 32^3
  // box 2.99 -> 2.78 ms)
  launch_k(k_body_apply, b.nb, sv.max_blobs > 20 ? 512 : 256, shm, s, b.nbl, b.boff, sv.shape_of, sv.off, sv.B,
           sv.offg, sv.G, b.quat, r, z, z64, d, b.st32, v);
  note_launch();
}

}  // namespace rbfib
