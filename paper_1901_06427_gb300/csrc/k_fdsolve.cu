// Exact solve of a coarse multigrid level by fast diagonalisation.  On a
// uniform box level every grid of the projection preconditioner has a
// separable operator: a velocity component of -eta LL (Sec. III.A; the
// ghost-reflection rows at tangential walls, odd at a no-slip and even at a
// free-slip wall, and the Dirichlet rows at the wall-normal boundary faces)
// and the Neumann pressure operator -D G are
// Kronecker sums of 1D second differences, one per axis.  Their eigenvectors
// are sine / cosine / Fourier bases in closed form, so the level solve is
// three 1D transforms, a diagonal scaling and three transforms back, done in
// shared memory.  This is the coarsest solve of the V-cycles, and the whole
// of them on all but the largest grids; the bases are built on the host once
// per grid and checked against the explicit 1D matrices.
#include <algorithm>
#include <cmath>
#include <cstdlib>

#include "common.cuh"
#include "kernels.cuh"

namespace rbfib {
namespace {

// kGhost: odd ghost at both ends (no-slip walls); kNeumann: even ghost at
// both ends (free-slip walls, and the pressure); kGhostNeumann /
// kNeumannGhost: odd at the low end and even at the high end, or the reverse.
enum AxisKind { kDirichlet, kGhost, kNeumann, kPeriodic, kGhostNeumann, kNeumannGhost };

// Row j of the 1D second-difference matrix (times h^2) of one kind: diag on
// the diagonal and -1 at the neighbours lo and hi; a missing neighbour (-1)
// adds +1 to the diagonal (ghost = -self), nothing (Dirichlet boundary value 0)
// or -1 (Neumann, ghost = self); periodic rows wrap.
void axis_row(AxisKind kind, int m, int j, double& diag, int& lo, int& hi) {
  diag = 2.0;
  lo = j - 1;
  hi = j + 1 < m ? j + 1 : -1;
  if (kind == kPeriodic) {
    lo = (j + m - 1) % m;
    hi = (j + 1) % m;
    return;
  }
  auto end = [&](bool odd, bool even) { diag += odd ? 1.0 : (even ? -1.0 : 0.0); };
  if (lo < 0) end(kind == kGhost || kind == kGhostNeumann, kind == kNeumann || kind == kNeumannGhost);
  if (hi < 0) end(kind == kGhost || kind == kNeumannGhost, kind == kNeumann || kind == kGhostNeumann);
}

// Orthonormal eigenvectors Q[j * m + k] = q_k(j) and eigenvalues of the
// matrix above: DST-I (Dirichlet), DST-II (ghost), DCT-II (Neumann), DST-IV
// (odd low end, even high end), DCT-IV (the reverse), real Fourier
// (periodic).  lam_0 = 0 exactly for the Neumann and periodic kinds.
// Every entry is a sine at a whole multiple of 2 pi / period, so the sines are
// computed once each (a call of the library per entry made grid creation on a
// 384 x 96 x 12 channel four times as long).
void axis_basis(AxisKind kind, int m, std::vector<double>& Q, std::vector<double>& lam) {
  const double pi = 3.14159265358979323846;
  Q.resize((size_t)m * m);
  lam.resize(m);
  const int period = kind == kDirichlet ? 2 * (m + 1) : (kind == kGhostNeumann || kind == kNeumannGhost ? 8 * m : 4 * m);
  std::vector<double> sine(period), scale(m);
  std::vector<int> at(m), step(m);
  for (int t = 0; t < period; ++t) sine[t] = std::sin(2.0 * pi * t / period);
  // column k at row j: scale * sine of (at + j step) / period turns
  for (int k = 0; k < m; ++k) {
    double th = 0.0;
    const int r = (k + 1) / 2;   // periodic: constant; cos / sin pairs of frequency r; (-1)^j for even m
    switch (kind) {
      case kDirichlet:     // sin(th (j + 1))
        th = pi * (k + 1) / (m + 1);
        scale[k] = std::sqrt(2.0 / (m + 1));
        at[k] = step[k] = k + 1;
        break;
      case kGhost:         // sin(th (j + 1/2))
        th = pi * (k + 1) / m;
        scale[k] = std::sqrt((k == m - 1 ? 1.0 : 2.0) / m);
        at[k] = k + 1;
        step[k] = 2 * (k + 1);
        break;
      case kNeumann:       // cos(th (j + 1/2))
        th = pi * k / m;
        scale[k] = std::sqrt((k == 0 ? 1.0 : 2.0) / m);
        at[k] = k + m;
        step[k] = 2 * k;
        break;
      case kGhostNeumann:  // sin(th (j + 1/2))
      case kNeumannGhost:  // cos(th (j + 1/2))
        th = pi * (k + 0.5) / m;
        scale[k] = std::sqrt(2.0 / m);
        at[k] = 2 * k + 1 + (kind == kNeumannGhost ? 2 * m : 0);
        step[k] = 2 * (2 * k + 1);
        break;
      case kPeriodic:      // cos(th j), sin(th j)
        th = 2.0 * pi * r / m;
        scale[k] = std::sqrt((k == 0 || 2 * r == m ? 1.0 : 2.0) / m);
        at[k] = k == 0 || (k & 1) ? m : 0;
        step[k] = 4 * r;
        break;
    }
    lam[k] = (k == 0 && (kind == kNeumann || kind == kPeriodic)) ? 0.0 : 2.0 - 2.0 * std::cos(th);
  }
  for (int j = 0; j < m; ++j)
    for (int k = 0; k < m; ++k) {
      Q[(size_t)j * m + k] = scale[k] * sine[at[k]];
      at[k] += step[k];
      if (at[k] >= period) at[k] -= period;
    }
}

// |T Q - Q diag(lam)| and the columns' norms, and the products of
// neighbouring columns.  T is symmetric with distinct eigenvalues but for
// the cos / sin pairs of a periodic axis, which are neighbours, so columns
// that pass are orthonormal.
bool basis_ok(AxisKind kind, int m, const std::vector<double>& Q, const std::vector<double>& lam) {
  const std::vector<double> none(m, 0.0);
  std::vector<double> res(m, 0.0), norm(m, 0.0), next(m, 0.0);
  for (int i = 0; i < m; ++i) {
    double diag;
    int lo, hi;
    axis_row(kind, m, i, diag, lo, hi);
    const double* q = &Q[(size_t)i * m];
    const double* ql = lo >= 0 ? &Q[(size_t)lo * m] : none.data();
    const double* qh = hi >= 0 ? &Q[(size_t)hi * m] : none.data();
    for (int k = 0; k < m; ++k) {
      res[k] = std::max(res[k], std::fabs((diag - lam[k]) * q[k] - ql[k] - qh[k]));
      norm[k] += q[k] * q[k];
    }
    for (int k = 0; k + 1 < m; ++k) next[k] += q[k] * q[k + 1];
  }
  double e1 = 0.0, e2 = 0.0;
  for (int k = 0; k < m; ++k) {
    e1 = std::max(e1, res[k]);
    e2 = std::max(e2, std::max(std::fabs(norm[k] - 1.0), std::fabs(next[k])));
  }
  return e1 <= 1e-12 * 4.0 * m && e2 <= 1e-13 * m;
}

// Basis rows in the table are padded to a multiple of 8 floats (zeros), so
// that chunks of outputs read whole 16-byte words inside their row.
RBFIB_DEVFN int fd_pad(int e) { return (e + 7) & ~7; }

// ------------------------------------------------------------------------
// Short lines (up to kFDLine points per axis), in three launches over the
// whole GPU: the forward x and y transforms of every z-plane, the z
// transform, eigenvalue scaling and backward z transform of every column, and
// the backward y and x transforms of every plane.  The level arrays stay in
// L2 between the launches.  Latency-bound: what counts is the chain load ->
// product -> product -> store of one block, so the products are blocked for
// few shared-memory reads per FMA and the basis tables, which no kernel
// writes, are staged before the wait on the preceding launch.
//
// One plane takes kFWX columns x kFWY groups of four rows of threads; the
// plane's output columns split over independent blocks.
constexpr int kFWX = 16, kFWY = kFDLine / 4, kFWThreads = kFWX * kFWY;
static_assert(4 * kFWY == kFDLine, "four rows per thread cover a line");

RBFIB_DEVFN int fd_planes(const FDGrid& G) { return G.e[2]; }
RBFIB_DEVFN int fd_col_tiles(const FDGrid& G) { return (G.e[0] * G.e[1] + 31) / 32; }

// Block index -> (grid gi, item k within the grid), items counted by f.
template <int (*F)(const FDGrid&)>
RBFIB_DEVFN void fd_item(const FDParams& P, int& k, int& gi) {
  gi = 0;
  while (gi < P.ng - 1 && k >= F(P.g[gi])) { k -= F(P.g[gi]); ++gi; }
}

// cp.async helpers: 16-byte and 4-byte global -> shared copies, one wait.
RBFIB_DEVFN void fdw_cp16(void* dst, const void* src) {
  asm volatile("cp.async.cg.shared.global [%0], [%1], 16;\n" ::"r"((unsigned)__cvta_generic_to_shared(dst)),
               "l"(src) : "memory");
}
RBFIB_DEVFN void fdw_cp4(void* dst, const void* src) {
  asm volatile("cp.async.ca.shared.global [%0], [%1], 4;\n" ::"r"((unsigned)__cvta_generic_to_shared(dst)),
               "l"(src) : "memory");
}
RBFIB_DEVFN void fdw_wait() {
  asm volatile("cp.async.commit_group;\n" ::: "memory");
  asm volatile("cp.async.wait_all;\n" ::: "memory");
}

// Stages the first e columns of the e rows of a basis table (rows padded to
// fd_pad(e) floats with zeros, 16-byte aligned) into M[kFDLine][kFDLine] by
// 16-byte copies.
RBFIB_DEVFN void fdw_stage_basis(float (*M)[kFDLine], const float* tab, int e) {
  const int ep = fd_pad(e), wpr = (e + 3) >> 2;
  for (int t = threadIdx.x; t < e * wpr; t += blockDim.x) {
    const int r = t / wpr, w = t - r * wpr;
    fdw_cp16(&M[r][4 * w], tab + r * ep + 4 * w);
  }
}

// One plane, one chunk of kFWX output columns (blockIdx.y): out = A_y (in
// A_x), the 1D transforms along x then y, with the forward bases (dir 0) or
// their transposes (dir 1).  Both transforms keep the output column: column
// c of A_x acts on the rows of the plane, and the y transform mixes rows of
// the same column.  The plane is staged transposed, so that a thread's four
// rows are one 16-byte word in both products: two shared-memory reads per
// four FMAs.  Velocity grids of 48 x 48 x 32 (285 blocks): 7.5 -> 6.3 us a
// launch against three rows per thread read one by one.
__global__ void __launch_bounds__(kFWThreads) k_fdw_xy(FDParams P, const float* __restrict__ in,
                                                       float* __restrict__ out, int dir) {
  __shared__ __align__(16) float XT[kFDLine][kFDLine + 4];
  __shared__ float T[kFDLine][kFWX + 4];
  __shared__ __align__(16) float Mx[kFDLine][kFWX];
  __shared__ __align__(16) float My[kFDLine][kFDLine];
  int k = blockIdx.x, gi;
  fd_item<fd_planes>(P, k, gi);
  const FDGrid& G = P.g[gi];
  const int e0 = G.e[0], e1 = G.e[1], p0 = fd_pad(e0), p1 = fd_pad(e1);
  const int c0 = blockIdx.y * kFWX;
  if (c0 >= e0) return;
  const float* Q0 = P.tab + G.tab0;
  const float* QT0 = Q0 + e0 * p0;
  const float* Q1 = QT0 + e0 * p0 + p0;
  const float* QT1 = Q1 + e1 * p1;
  const float* ax = dir ? QT0 : Q0;
  const int tx = threadIdx.x % kFWX, ty = threadIdx.x / kFWX;
  // the chunk's columns of A_x (rows padded to 8 floats, so the 16 columns
  // from c0 are four whole 16-byte words inside the row) and A_y
  for (int t = threadIdx.x; t < e0 * (kFWX / 4); t += kFWThreads) {
    const int r = t / (kFWX / 4), w = t - r * (kFWX / 4);
    if (c0 + 4 * w < p0) fdw_cp16(&Mx[r][4 * w], ax + r * p0 + c0 + 4 * w);
  }
  fdw_stage_basis(My, dir ? QT1 : Q1, e1);
  pdl_entry();
  const float* src = in + G.off + (long long)k * e0 * e1;
  for (int r = threadIdx.x >> 5; r < e1; r += kFWThreads / 32)
    for (int c = threadIdx.x & 31; c < e0; c += 32) fdw_cp4(&XT[c][r], src + r * e0 + c);
  fdw_wait();
  __syncthreads();
  // T[j][c] = sum_i X[j][i] A_x[i][c0 + c]  (rows j >= e1 are never read back)
  float acc[4] = {0.f, 0.f, 0.f, 0.f};
#pragma unroll 8
  for (int i = 0; i < e0; ++i) {
    const float m = Mx[i][tx];
    const float4 x = *reinterpret_cast<const float4*>(&XT[i][4 * ty]);
    acc[0] = fmaf(x.x, m, acc[0]);
    acc[1] = fmaf(x.y, m, acc[1]);
    acc[2] = fmaf(x.z, m, acc[2]);
    acc[3] = fmaf(x.w, m, acc[3]);
  }
#pragma unroll
  for (int a = 0; a < 4; ++a) {
    T[4 * ty + a][tx] = acc[a];
    acc[a] = 0.f;
  }
  __syncthreads();
  // out[r][c] = sum_j A_y[j][r] T[j][c]
#pragma unroll 8
  for (int j = 0; j < e1; ++j) {
    const float t = T[j][tx];
    const float4 m = *reinterpret_cast<const float4*>(&My[j][4 * ty]);
    acc[0] = fmaf(m.x, t, acc[0]);
    acc[1] = fmaf(m.y, t, acc[1]);
    acc[2] = fmaf(m.z, t, acc[2]);
    acc[3] = fmaf(m.w, t, acc[3]);
  }
  float* dst = out + G.off + (long long)k * e0 * e1;
  const int c = c0 + tx;
#pragma unroll
  for (int a = 0; a < 4; ++a) {
    const int r = 4 * ty + a;
    if (r < e1 && c < e0) dst[r * e0 + c] = acc[a];
  }
}

// 32 adjacent columns (fixed x, y; all z) of one grid, in place: forward z
// transform, division by s (l_x + l_y + l_z) (the zero mode of a singular
// grid dropped), backward z transform.  Thread (column ci, group gr) holds
// its whole column in registers and forms the outputs gr, gr + 8, ...: per
// four FMAs one broadcast 16-byte read of the basis row (a column read again
// for every output took two reads per FMA: 9.6 -> 7.2 us at 48 x 48 x 32).
// Levels of up to 32^3 points ran on one cluster per grid before; the three
// launches take one sphere's mobility solve in a 32^3 box from 5.5 to 3.5 ms.
__global__ void __launch_bounds__(256) k_fdw_z(FDParams P, float* __restrict__ data) {
  __shared__ float Z[kFDLine][33];
  __shared__ __align__(16) float Mz[kFDLine][kFDLine];
  __shared__ __align__(16) float MzT[kFDLine][kFDLine];
  int tile = blockIdx.x, gi;
  fd_item<fd_col_tiles>(P, tile, gi);
  const FDGrid& G = P.g[gi];
  const int e0 = G.e[0], e1 = G.e[1], e2 = G.e[2], pl = e0 * e1;
  const float* L0 = P.tab + G.lam[0];
  const float* L1 = P.tab + G.lam[1];
  const float* L2 = P.tab + G.lam[2];
  fdw_stage_basis(Mz, P.tab + G.q2, e2);
  fdw_stage_basis(MzT, P.tab + G.qt2, e2);
  const int ci = threadIdx.x & 31, gr = threadIdx.x >> 5;
  const int col = tile * 32 + ci;
  const bool live = col < pl;
  const float sxy = live ? L0[col % e0] + L1[col / e0] : 0.f;
  pdl_entry();
  float* base = data + G.off;
  if (live)
    for (int kk = gr; kk < e2; kk += 8) fdw_cp4(&Z[kk][ci], base + (long long)kk * pl + col);
  fdw_wait();
  __syncthreads();
  float z[kFDLine];
  auto column = [&]() {
#pragma unroll
    for (int kk = 0; kk < kFDLine; ++kk) z[kk] = kk < e2 ? Z[kk][ci] : 0.f;
  };
  // sum_k M[row][k] z[k]; M's row is zero-padded to a multiple of four
  auto dot = [&](const float (*M)[kFDLine], int row) {
    float a[4] = {0.f, 0.f, 0.f, 0.f};
#pragma unroll
    for (int b = 0; b < kFDLine / 4; ++b) {
      if (4 * b < e2) {
        const float4 m = *reinterpret_cast<const float4*>(&M[row][4 * b]);
        a[0] = fmaf(m.x, z[4 * b], a[0]);
        a[1] = fmaf(m.y, z[4 * b + 1], a[1]);
        a[2] = fmaf(m.z, z[4 * b + 2], a[2]);
        a[3] = fmaf(m.w, z[4 * b + 3], a[3]);
      }
    }
    return (a[0] + a[1]) + (a[2] + a[3]);
  };
  column();
  __syncthreads();
  for (int c = gr; c < e2; c += 8) {
    const float s = G.scale * (sxy + L2[c]);
    const float t = dot(MzT, c);
    Z[c][ci] = s > 0.f ? t / s : 0.f;
  }
  __syncthreads();
  column();
  for (int kk = gr; kk < e2; kk += 8) {
    const float t = dot(Mz, kk);
    if (live) base[(long long)kk * pl + col] = t;
  }
}

// ------------------------------------------------------------------------
// Long lines: levels with an axis of more than kFDLine points.  Each axis is
// one pass over the level, a batch of small products line x basis, tiled as
// matrix products over the whole GPU (x, y, z forward, then z, y, x back; a
// z axis of at most kFDLine points takes k_fdw_z instead of its two passes).
//
// The eigenvectors of every axis kind but the mixed free-slip / no-slip ones
// are even or odd under the mirror j -> m - 1 - j (periodic axes: j -> -j),
// so a line is folded into sums and differences of mirrored points and the
// even and odd eigenvectors each see half of it: half the products of the
// plain basis.  Pair p of an axis joins points a and b (a == b: its own
// mirror, no odd part).
//
// Bound by the FP32 pipe and by latency on small levels.  It takes the place
// of the V-cycles above a short-line level (28 launches at their launch floor
// on the 384 x 96 x 12 channel, whose flat levels point smoothing treats
// badly): driven monolayer step 299 -> 177 ms (704 -> 399 iterations),
// 128 x 128 x 64 gradient 365 -> 104 ms (about 600 -> 230), boomerang slit
// step 18.4 -> 14.0 ms.
// b = sum - p, but for the points that are their own mirror (fold_sum; the
// point 0 of a periodic axis, every point without a mirror).
RBFIB_DEVFN int fold_sum(const FDAxis& X) { return X.fold == kFoldMirror ? X.e - 1 : (X.fold == kFoldPeriodic ? X.e : -1); }
RBFIB_DEVFN int fold_partner(int sum, int e, int p) { const int b = sum - p; return sum < 0 || b >= e ? p : b; }

// Shape of a pass: 128 threads, 64 entries along the contiguous dimension of
// memory (16 threads x 4 interleaved, so that stores of a warp are
// contiguous) by 8 TM of the other one (8 threads x TM), kFLK steps of the
// product per stage.  AX = 0: lines along x, whose contiguous dimension is
// the line itself; AX = 1: lines along y or z, adjacent lines contiguous.
// TM = 8 needs 6 shared-memory wavefronts for the 8 cycles that a warp's 32
// FMAs take (TM = 4: 5 for 4), so it is used where it leaves enough blocks.
constexpr int kFLThreads = 128, kFLC = 64, kFLK = 16;

// Line l of the axis: offset of its first point; stride along the axis.
RBFIB_DEVFN int fdl_base(const FDGrid& G, int axis, int l) {
  if (axis == 0) return l * G.e[0];
  if (axis == 1) {
    const int z = l / G.e[0];
    return (l - z * G.e[0]) + z * G.e[0] * G.e[1];
  }
  return l;
}
RBFIB_DEVFN int fdl_stride(const FDGrid& G, int axis) { return axis == 0 ? 1 : (axis == 1 ? G.e[0] : G.e[0] * G.e[1]); }

template <int AX, int TM>
struct FdlTile {
  static constexpr int LT = AX == 0 ? 8 * TM : kFLC;   // lines
  static constexpr int CT = AX == 0 ? kFLC : 8 * TM;   // outputs along the axis
  static constexpr int FN = kFLK * LT / kFLThreads;    // staged line entries of a thread
  static constexpr int BN = kFLK * CT / 4 / kFLThreads > 0 ? kFLK * CT / 4 / kFLThreads : 1;   // staged float4 of the basis
  float F[2][kFLK][LT + 4];
  float B[2][kFLK][CT + 4];
};

// acc += F B over one stage
template <int AX, int TM>
RBFIB_DEVFN void fdl_fma(const FdlTile<AX, TM>& S, int buf, int tx, int ty, float acc[TM][4]) {
#pragma unroll
  for (int k = 0; k < kFLK; ++k) {
    const float* co = AX == 0 ? S.B[buf][k] : S.F[buf][k];
    const float* ot = AX == 0 ? S.F[buf][k] : S.B[buf][k];
    float o[TM], c[4];
#pragma unroll
    for (int q = 0; q < TM / 4; ++q) {
      const float4 v = *reinterpret_cast<const float4*>(ot + TM * ty + 4 * q);
      o[4 * q] = v.x; o[4 * q + 1] = v.y; o[4 * q + 2] = v.z; o[4 * q + 3] = v.w;
    }
#pragma unroll
    for (int i = 0; i < 4; ++i) c[i] = co[tx + 16 * i];
#pragma unroll
    for (int r = 0; r < TM; ++r)
#pragma unroll
      for (int i = 0; i < 4; ++i) acc[r][i] = fmaf(o[r], c[i], acc[r][i]);
  }
}

// The product of K steps: load(k, line) gives the line entry of step k,
// B (rows of pitch floats) the basis from column c0.
template <int AX, int TM, typename Load>
RBFIB_DEVFN void fdl_product(FdlTile<AX, TM>& S, int K, const float* __restrict__ B, int pitch, int c0, Load load,
                             float acc[TM][4]) {
  typedef FdlTile<AX, TM> Tl;
  const int t = threadIdx.x, tx = t & 15, ty = t >> 4;
  float rf[Tl::FN];
  float4 rb[Tl::BN];
  auto fetch = [&](int k0) {
#pragma unroll
    for (int i = 0; i < Tl::FN; ++i) {
      const int e = t + kFLThreads * i;
      const int kk = AX == 0 ? e % kFLK : e / Tl::LT, l = AX == 0 ? e / kFLK : e % Tl::LT;
      rf[i] = load(min(k0 + kk, K - 1), l);   // past K the basis rows are zero
    }
#pragma unroll
    for (int i = 0; i < Tl::BN; ++i) {
      const int e = t + kFLThreads * i;
      const int kk = e / (Tl::CT / 4), c = c0 + 4 * (e % (Tl::CT / 4));
      rb[i] = (kk < kFLK && k0 + kk < K && c < pitch)
                  ? __ldg(reinterpret_cast<const float4*>(B + (long long)(k0 + kk) * pitch + c))
                  : make_float4(0.f, 0.f, 0.f, 0.f);
    }
  };
  auto put = [&](int buf) {
#pragma unroll
    for (int i = 0; i < Tl::FN; ++i) {
      const int e = t + kFLThreads * i;
      const int kk = AX == 0 ? e % kFLK : e / Tl::LT, l = AX == 0 ? e / kFLK : e % Tl::LT;
      S.F[buf][kk][l] = rf[i];
    }
#pragma unroll
    for (int i = 0; i < Tl::BN; ++i) {
      const int e = t + kFLThreads * i;
      const int kk = e / (Tl::CT / 4);
      if (kk < kFLK) *reinterpret_cast<float4*>(&S.B[buf][kk][4 * (e % (Tl::CT / 4))]) = rb[i];
    }
  };
  fetch(0);
  put(0);
  __syncthreads();
  int buf = 0;
  for (int k0 = 0; k0 < K; k0 += kFLK) {
    const bool more = k0 + kFLK < K;
    if (more) fetch(k0 + kFLK);
    fdl_fma<AX, TM>(S, buf, tx, ty, acc);
    if (more) put(buf ^ 1);
    __syncthreads();
    buf ^= 1;
  }
}

// Forward transform along one axis: blockIdx.x line tiles, blockIdx.y tiles
// of the even, then of the odd eigenvectors, blockIdx.z grids.  scaled: the
// last forward pass divides by s (l_x + l_y + l_z) (z axis; zero modes
// dropped).
template <int AX, int TM>
__global__ void __launch_bounds__(kFLThreads) k_fdl_fwd(FDParams P, int axis, int scaled,
                                                        const float* __restrict__ in, float* __restrict__ out) {
  pdl_entry();
  typedef FdlTile<AX, TM> Tl;
  __shared__ __align__(16) Tl S;
  const FDGrid& G = P.g[blockIdx.z];
  // in registers: a read of the parameters by a run-time index per staged
  // entry would stall each one
  const FDAxis X = G.ax[axis];
  const int e0 = G.e[0], nl = e0 * G.e[1] * G.e[2] / X.e, l0 = blockIdx.x * Tl::LT, sum = fold_sum(X);
  const int nS = (X.hs + Tl::CT - 1) / Tl::CT, nA = (X.ha + Tl::CT - 1) / Tl::CT;
  if (l0 >= nl || (int)blockIdx.y >= nS + nA) return;
  const bool odd = (int)blockIdx.y >= nS;
  const int c0 = ((int)blockIdx.y - (odd ? nS : 0)) * Tl::CT, nc = odd ? X.ha : X.hs;
  const float* src = in + G.off;
  const int st = fdl_stride(G, axis);
  float acc[TM][4];
#pragma unroll
  for (int r = 0; r < TM; ++r)
#pragma unroll
    for (int i = 0; i < 4; ++i) acc[r][i] = 0.f;
  const int last = nl - 1;
  const float sg = odd ? -1.f : 1.f;
  // AX = 1: the lines of a thread's entries are the same in every stage
  const int own = AX == 1 ? fdl_base(G, axis, min(l0 + (int)threadIdx.x % Tl::LT, last)) : 0;
  fdl_product<AX, TM>(
      S, X.hs, P.tab + (odd ? X.fA : X.fS), odd ? X.pa : X.ps, c0,
      [&](int p, int l) {
        const int b = fold_partner(sum, X.e, p);
        const float* line = src + (AX == 1 ? own : min(l0 + l, last) * e0);
        // both points loaded without a branch, so that a stage's loads are in
        // flight together
        const float va = line[p * st], vb = line[b * st];
        return fmaf(p == b ? 0.f : sg, vb, va);
      },
      acc);
  const int tx = threadIdx.x & 15, ty = threadIdx.x >> 4;
  float* dst = out + G.off;
  const int shift = odd ? X.hs : 0;
#pragma unroll
  for (int r = 0; r < TM; ++r)
#pragma unroll
    for (int i = 0; i < 4; ++i) {
      const int co = tx + 16 * i, ot = TM * ty + r;
      const int l = l0 + (AX == 0 ? ot : co), c = c0 + (AX == 0 ? co : ot);
      if (l >= nl || c >= nc) continue;
      float v = acc[r][i];
      if (scaled) {
        const int y = l / G.e[0];
        const float s = G.scale * ((P.tab[G.lam[0] + l - y * G.e[0]] + P.tab[G.lam[1] + y]) + P.tab[G.lam[2] + shift + c]);
        v = s > 0.f ? v / s : 0.f;
      }
      dst[fdl_base(G, axis, l) + (shift + c) * st] = v;
    }
}

// Backward transform along one axis: the even and the odd part of a pair
// are summed apart, then the pair's two points are their sum and difference.
template <int AX, int TM>
__global__ void __launch_bounds__(kFLThreads) k_fdl_bwd(FDParams P, int axis, const float* __restrict__ in,
                                                        float* __restrict__ out) {
  pdl_entry();
  typedef FdlTile<AX, TM> Tl;
  __shared__ __align__(16) Tl S;
  const FDGrid& G = P.g[blockIdx.z];
  const FDAxis X = G.ax[axis];
  const int e0 = G.e[0], nl = e0 * G.e[1] * G.e[2] / X.e, l0 = blockIdx.x * Tl::LT, p0 = blockIdx.y * Tl::CT;
  if (l0 >= nl || p0 >= X.hs) return;
  const float* src = in + G.off;
  const int st = fdl_stride(G, axis), last = nl - 1;
  const int own = AX == 1 ? fdl_base(G, axis, min(l0 + (int)threadIdx.x % Tl::LT, last)) : 0;
  float ev[TM][4], od[TM][4];
#pragma unroll
  for (int r = 0; r < TM; ++r)
#pragma unroll
    for (int i = 0; i < 4; ++i) { ev[r][i] = 0.f; od[r][i] = 0.f; }
  fdl_product<AX, TM>(
      S, X.hs, P.tab + X.bS, X.ps, p0,
      [&](int c, int l) { return src[(AX == 1 ? own : min(l0 + l, last) * e0) + c * st]; }, ev);
  if (X.ha > 0)
    fdl_product<AX, TM>(
        S, X.ha, P.tab + X.bA, X.ps, p0,
        [&](int c, int l) { return src[(AX == 1 ? own : min(l0 + l, last) * e0) + (X.hs + c) * st]; }, od);
  const int tx = threadIdx.x & 15, ty = threadIdx.x >> 4, sum = fold_sum(X);
  float* dst = out + G.off;
#pragma unroll
  for (int r = 0; r < TM; ++r)
#pragma unroll
    for (int i = 0; i < 4; ++i) {
      const int co = tx + 16 * i, ot = TM * ty + r;
      const int l = l0 + (AX == 0 ? ot : co), p = p0 + (AX == 0 ? co : ot);
      if (l >= nl || p >= X.hs) continue;
      const int b = fold_partner(sum, X.e, p);
      float* line = dst + fdl_base(G, axis, l);
      line[p * st] = ev[r][i] + od[r][i];
      if (p != b) line[b * st] = ev[r][i] - od[r][i];
    }
}

template <int AX, int TM>
void fdl_launch(const FDParams& P, int axis, bool fwd, int scaled, const float* in, float* out, cudaStream_t s) {
  typedef FdlTile<AX, TM> Tl;
  int gx = 1, gy = 1;
  for (int g = 0; g < P.ng; ++g) {
    const FDAxis& X = P.g[g].ax[axis];
    const int nl = P.g[g].e[0] * P.g[g].e[1] * P.g[g].e[2] / X.e;
    gx = std::max(gx, (nl + Tl::LT - 1) / Tl::LT);
    gy = std::max(gy, (X.hs + Tl::CT - 1) / Tl::CT + (fwd ? (X.ha + Tl::CT - 1) / Tl::CT : 0));
  }
  if (fwd) launch_k(k_fdl_fwd<AX, TM>, dim3(gx, gy, P.ng), kFLThreads, 0, s, P, axis, scaled, in, out);
  else launch_k(k_fdl_bwd<AX, TM>, dim3(gx, gy, P.ng), kFLThreads, 0, s, P, axis, in, out);
  note_launch();
}

// One pass, with the wide tile where that still gives two blocks per SM.
void fdl_pass(const FDParams& P, int axis, bool fwd, int scaled, const float* in, float* out, cudaStream_t s) {
  long long tiles = 0;
  for (int g = 0; g < P.ng; ++g) {
    const FDAxis& X = P.g[g].ax[axis];
    const long long nl = (long long)P.g[g].e[0] * P.g[g].e[1] * P.g[g].e[2] / X.e;
    tiles += ((nl + 63) / 64) * ((X.hs + 63) / 64 + (fwd ? (X.ha + 63) / 64 : 0));
  }
  const bool big = tiles >= 2 * 152;
  if (axis == 0) {
    if (big) fdl_launch<0, 8>(P, axis, fwd, scaled, in, out, s);
    else fdl_launch<0, 4>(P, axis, fwd, scaled, in, out, s);
  } else {
    if (big) fdl_launch<1, 8>(P, axis, fwd, scaled, in, out, s);
    else fdl_launch<1, 4>(P, axis, fwd, scaled, in, out, s);
  }
}

void fd_solve_lines(const FDParams& P, float* u, const float* rhs, float* tmp, cudaStream_t s) {
  fdl_pass(P, 0, true, 0, rhs, tmp, s);
  fdl_pass(P, 1, true, 0, tmp, u, s);
  if (P.g[0].q2) {
    int tiles = 0;
    for (int g = 0; g < P.ng; ++g) tiles += (P.g[g].e[0] * P.g[g].e[1] + 31) / 32;
    launch_k(k_fdw_z, tiles, 256, 0, s, P, u);
    note_launch();
  } else {
    fdl_pass(P, 2, true, 1, u, tmp, s);
    fdl_pass(P, 2, false, 0, tmp, u, s);
  }
  fdl_pass(P, 1, false, 0, u, tmp, s);
  fdl_pass(P, 0, false, 0, tmp, u, s);
}

void fd_solve_short(const FDParams& P, float* u, const float* rhs, float* tmp, cudaStream_t s) {
  int planes = 0, tiles = 0, chunks = 1;
  for (int g = 0; g < P.ng; ++g) {
    planes += P.g[g].e[2];
    tiles += (P.g[g].e[0] * P.g[g].e[1] + 31) / 32;
    chunks = std::max(chunks, (P.g[g].e[0] + kFWX - 1) / kFWX);
  }
  launch_k(k_fdw_xy, dim3(planes, chunks), kFWThreads, 0, s, P, rhs, tmp, 0);
  note_launch();
  launch_k(k_fdw_z, tiles, 256, 0, s, P, tmp);
  note_launch();
  launch_k(k_fdw_xy, dim3(planes, chunks), kFWThreads, 0, s, P, (const float*)tmp, u, 1);
  note_launch();
}

}  // namespace

// Longest line of the short-line form: kFDLine, or a smaller value from
// RBFIB_FD_LINE (read once).
static int fd_line_limit() {
  static const int lim = [] {
    const char* e = std::getenv("RBFIB_FD_LINE");
    const int v = e ? std::atoi(e) : kFDLine;
    return (v >= 1 && v <= kFDLine) ? v : kFDLine;
  }();
  return lim;
}

// Largest e_x + e_y + e_z solved in the long-line form; RBFIB_FD_SUM
// overrides it (read once; 0 measures the V-cycles).  The exact solve costs
// 2 (e_x + e_y + e_z) operations per point and direction, the V-cycles above
// a short-line level a fixed number of passes and launches, and the exact
// solve saves iterations.  Stokes solves to 1e-8 (FP32 refined), exact
// against V-cycles: 96^3 8.9 / 11.2 ms, 160^3 40.5 / 42.1, 192^3 64.9 /
// 69.7, 256^3 152 / 172; larger grids keep the V-cycles on their finest levels.
constexpr int kFDLinesSum = 800;
static int fd_lines_limit() {
  static const int lim = [] {
    const char* e = std::getenv("RBFIB_FD_SUM");
    return e ? std::atoi(e) : kFDLinesSum;
  }();
  return lim;
}

namespace {

AxisKind axis_kind(const Dims& d, bool faces, int g, int ax) {
  if (d.per[ax]) return kPeriodic;
  if (!faces) return kNeumann;
  if (ax == g) return kDirichlet;
  const bool even_lo = ghost_sign(d, 2 * ax) > 0, even_hi = ghost_sign(d, 2 * ax + 1) > 0;
  return even_lo ? (even_hi ? kNeumann : kNeumannGhost) : (even_hi ? kGhostNeumann : kGhost);
}

// Columns of the basis of kind even (odd = 0) or odd (1) under the mirror of
// the axis: every other one, starting with the even column 0; on periodic
// axes the constant and the cosines, then the sines; all of them, as even
// ones, where there is no mirror.
std::vector<int> fold_columns(AxisKind kind, int m, int odd) {
  std::vector<int> c;
  const bool none = kind == kGhostNeumann || kind == kNeumannGhost;
  for (int k = 0; k < m; ++k) {
    const bool is_odd = kind == kPeriodic ? (k > 0 && k % 2 == 0) : (!none && k % 2 == 1);
    if (is_odd == (odd != 0)) c.push_back(k);
  }
  return c;
}

// Appends the folded tables of one axis (FDAxis) and its eigenvalues in
// folded order.
void fold_axis(AxisKind kind, int m, const std::vector<double>& Q, const std::vector<double>& lam, double ih2,
               std::vector<float>& tab, FDAxis& X, int& lam0) {
  const std::vector<int> cs = fold_columns(kind, m, 0), ca = fold_columns(kind, m, 1);
  X.e = m;
  X.fold = kind == kPeriodic ? kFoldPeriodic : (kind == kGhostNeumann || kind == kNeumannGhost ? kFoldNone : kFoldMirror);
  X.hs = (int)cs.size();
  X.ha = (int)ca.size();
  X.ps = (X.hs + 3) & ~3;
  X.pa = (X.ha + 3) & ~3;
  auto self = [&](int p) {
    return X.fold == kFoldNone || (X.fold == kFoldMirror ? 2 * p == m - 1 : p == 0 || 2 * p == m);
  };
  auto zeros = [&](int nr, int pitch) {
    const int at = (int)tab.size();
    tab.resize(tab.size() + (size_t)nr * pitch, 0.f);
    return at;
  };
  X.fS = zeros(X.hs, X.ps);
  X.fA = zeros(X.hs, X.pa);
  X.bS = zeros(X.hs, X.ps);
  X.bA = zeros(X.ha, X.ps);
  for (int p = 0; p < X.hs; ++p) {
    const double* q = &Q[(size_t)p * m];
    for (int c = 0; c < X.hs; ++c)
      tab[X.fS + (size_t)p * X.ps + c] = tab[X.bS + (size_t)c * X.ps + p] = (float)q[cs[c]];
    if (!self(p))
      for (int c = 0; c < X.ha; ++c)
        tab[X.fA + (size_t)p * X.pa + c] = tab[X.bA + (size_t)c * X.ps + p] = (float)q[ca[c]];
  }
  lam0 = (int)tab.size();
  for (int k : cs) tab.push_back((float)(lam[k] * ih2));
  for (int k : ca) tab.push_back((float)(lam[k] * ih2));
  while (tab.size() % 4) tab.push_back(0.f);
}

// The basis in plain order: Q and Q^T (rows padded to 8 floats), then the
// eigenvalues.
void plain_axis(int m, const std::vector<double>& Q, const std::vector<double>& lam, double ih2,
                std::vector<float>& tab, int& q0, int& qt0, int& lam0) {
  const int mp = (m + 7) & ~7;
  q0 = (int)tab.size();
  qt0 = q0 + m * mp;
  tab.resize(tab.size() + 2 * (size_t)m * mp, 0.f);
  for (int t = 0; t < m; ++t)
    for (int c = 0; c < m; ++c) tab[q0 + t * mp + c] = tab[qt0 + c * mp + t] = (float)Q[(size_t)t * m + c];
  lam0 = (int)tab.size();
  for (int c = 0; c < mp; ++c) tab.push_back(c < m ? (float)(lam[c] * ih2) : 0.f);
}

}  // namespace

bool fd_plan(const Dims& d, bool faces, double eta, std::vector<float>& tab, FDParams& P, std::string& why) {
  P = FDParams{};
  P.ng = faces ? 3 : 1;
  const size_t tab_start = tab.size();
  auto fail = [&](const char* w) { why = w; tab.resize(tab_start); return false; };
  int longest = 0, ez = 0, sum = 0;
  for (int g = 0; g < P.ng; ++g) {
    const int* e = faces ? d.fe[g] : d.n;
    for (int ax = 0; ax < 3; ++ax) {
      if (e[ax] < 1) return fail("extent");
      longest = std::max(longest, e[ax]);
    }
    ez = std::max(ez, e[2]);
    sum = std::max(sum, e[0] + e[1] + e[2]);
  }
  P.lines = longest > fd_line_limit() ? 1 : 0;
  if (P.lines && (longest > kFDLongest || sum > fd_lines_limit() || d.fo[3] + d.nc >= (1LL << 31))) return fail("extent");
  // z-axis basis in plain order too, for k_fdw_z
  const bool plain_z = !P.lines || ez <= kFDLine;
  // grids of one level share most of their axes: bases, and in the long-line
  // form (no segment of its own per grid) their place in the table
  struct Basis { AxisKind kind; int m; std::vector<double> Q, lam; bool placed[2]; FDAxis ax; int lam0, q2, qt2, lam2; double ih2; };
  std::vector<Basis> seen;
  while (tab.size() % 4 || tab.empty()) tab.push_back(0.f);
  for (int g = 0; g < P.ng; ++g) {
    FDGrid& G = P.g[g];
    const int* e = faces ? d.fe[g] : d.n;
    G.off = faces ? d.fo[g] : 0;
    G.scale = faces ? (float)eta : 1.0f;
    G.tab0 = (int)tab.size();
    for (int ax = 0; ax < 3; ++ax) {
      const int m = G.e[ax] = e[ax];
      const AxisKind kind = axis_kind(d, faces, g, ax);
      const double ih2 = 1.0 / (d.h[ax] * d.h[ax]);
      Basis* B = nullptr;
      for (Basis& b : seen)
        if (b.kind == kind && b.m == m && b.ih2 == ih2) B = &b;
      if (!B) {
        seen.emplace_back();
        B = &seen.back();
        *B = Basis{kind, m, {}, {}, {false, false}, {}, 0, 0, 0, 0, ih2};
        axis_basis(kind, m, B->Q, B->lam);
        if (!basis_ok(kind, m, B->Q, B->lam)) return fail("basis check");
      }
      const bool plain = !P.lines || (ax == 2 && plain_z);
      if (!P.lines || !B->placed[plain]) {
        if (plain) plain_axis(m, B->Q, B->lam, ih2, tab, B->q2, B->qt2, B->lam2);
        else fold_axis(kind, m, B->Q, B->lam, ih2, tab, B->ax, B->lam0);
        B->placed[plain] = true;
      }
      if (plain) {
        G.lam[ax] = B->lam2;
        if (ax == 2) { G.q2 = B->q2; G.qt2 = B->qt2; }
        G.ax[ax].e = m;
      } else {
        G.ax[ax] = B->ax;
        G.lam[ax] = B->lam0;
      }
    }
    G.tabn = (int)tab.size() - G.tab0;
    // every grid's segment starts on a 16-byte boundary of the table
    while (tab.size() % 4) tab.push_back(0.f);
  }
  return true;
}

void fd_solve(const FDParams& P, float* u, const float* rhs, float* tmp, cudaStream_t s) {
  if (P.lines) fd_solve_lines(P, u, rhs, tmp, s);
  else fd_solve_short(P, u, rhs, tmp, s);
}

}  // namespace rbfib
