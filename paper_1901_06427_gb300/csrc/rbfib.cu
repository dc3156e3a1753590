// Host side of librbfib: the grid object, the multigrid hierarchy, the
// preconditioned FGMRES solver of the constrained saddle system (Sec. III.C),
// the Split-Euler-Maruyama step (Sec. IV.B, Algorithm 1) and the C ABI.
#include <algorithm>
#include <cmath>
#include <cstdio>
#include <cstdlib>
#include <cstring>
#include <map>
#include <mutex>
#include <string>
#include <type_traits>
#include <vector>

#include "../../include/rbfib.h"
#include "common.cuh"
#include "kernels.cuh"
#include "pair_mobility.cuh"

using namespace rbfib;

std::atomic<unsigned long long> rbfib::g_launches{0};

bool rbfib::pdl_enabled() {
  static const bool on = std::getenv("RBFIB_NO_PDL") == nullptr;
  return on;
}

namespace {

const double kDeltaDefault = 6.0554544523933395e-06;   // eps^(1/3), eps = 2^-52
const double kInnerTol = 1e-4;   // relative reduction asked of each FP32 refinement sweep
const int kDenseBodyMaxRows = 1536;                      // 3 N_bl limit of the coupled body block
const int kDenseBodyMaxBodyRows = 384;                   // 6 N_b limit of the coupled body block

// A failed CUDA runtime call, or (code other than RBFIB_ECUDA) an
// inconsistency found on the host after a device step, such as a singular
// pivot in the body block's set-up.
struct CudaError {
  cudaError_t e;
  int code = RBFIB_ECUDA;
  const char* msg = nullptr;
  const char* what() const { return msg ? msg : cudaGetErrorString(e); }
};

inline void ck(cudaError_t e) {
  if (e != cudaSuccess) throw CudaError{e};
}

template <typename T>
struct DBuf {
  T* p = nullptr;
  size_t n = 0;
  DBuf() = default;
  DBuf(const DBuf&) = delete;
  DBuf& operator=(const DBuf&) = delete;
  void alloc(size_t k) {
    release();
    if (k) ck(cudaMalloc((void**)&p, k * sizeof(T)));
    n = k;
  }
  void ensure(size_t k) {
    if (k > n) alloc(k);
  }
  void release() {
    if (p) cudaFree(p);
    p = nullptr;
    n = 0;
  }
  ~DBuf() { release(); }
  operator T*() const { return p; }
};

struct Level {
  Dims d;
  int3 cz;   // axes coarsened towards the next level
};

// Multigrid storage of one precision.
template <typename T>
struct MGStore {
  std::vector<DBuf<T>*> vu, vrhs, vres, pu, prhs, pres;
  void build(const std::vector<Level>& L) {
    release();
    for (size_t l = 0; l < L.size(); ++l) {
      const i64 nf = L[l].d.fo[3], nc = L[l].d.nc;
      auto mk = [](i64 n) { auto* b = new DBuf<T>(); b->alloc(n); return b; };
      vu.push_back(mk(nf)); vrhs.push_back(mk(nf)); vres.push_back(mk(nf));
      pu.push_back(mk(nc)); prhs.push_back(mk(nc)); pres.push_back(mk(nc));
    }
  }
  void release() {
    for (auto* v : {&vu, &vrhs, &vres, &pu, &prhs, &pres}) {
      for (auto* b : *v) delete b;
      v->clear();
    }
  }
  ~MGStore() { release(); }
};

// Krylov storage of one precision (basis V, flexible basis Z).
template <typename T>
struct KrylovStore {
  int m = 0;
  i64 n = 0;
  DBuf<T> V, Z, w;
  // captured iterations: FP32 copy of the newest basis vector and the
  // preconditioned vector
  DBuf<float> v32;
  DBuf<T> z;
  void build(int m_, i64 n_) {
    // columns start on 32-byte boundaries (16-byte vector loads in FP64 and FP32)
    const i64 ld = (n_ + 3) & ~(i64)3;
    n = 0;   // until all of it is there
    m = m_;
    V.alloc((size_t)(m + 1) * ld);
    Z.alloc((size_t)m * ld);
    w.alloc(ld);
    v32.alloc(ld);
    z.alloc(ld);
    n = ld;
  }
};

struct Config {   // one body configuration (positions derived from q, quat)
  DBuf<double> q, quat, r, arm;
  DBuf<int> perm;
  DBuf<BlobStencil<double>> st64;   // kernel stencils (current configuration only)
  DBuf<BlobStencil<float>> st32;
};

}  // namespace

// Threads per block of the finest-level stencil and smoothing kernels, picked
// by timing candidates once per grid shape (see autotune).
struct Tuning {
  int stokes64 = 256, stokes32 = 256, vrbgs = 256, prbgs = 256;
};

struct rbfib_grid {
  Tuning tune;
  rbfib_grid_desc desc{};
  cudaStream_t s = nullptr;
  std::string err;
  std::vector<Level> levels;
  int fd_vel = -1, fd_p = -1;   // levels solved exactly by fast diagonalisation (-1: none)
  FDParams fdv{}, fdp{};
  DBuf<float> fd_tab, fd_tmp;
  Dims d{};
  Walls walls{};
  bool walls_move = false;   // some wall velocity is not zero
  i64 nf = 0, nc = 0, nfl = 0;
  double dV = 1.0;
  double kappa = 0.0;   // pressure_kappa
  StressLayout stress{};
  // bodies
  int nb = 0, nbl = 0;
  std::vector<int> h_boff;
  DBuf<int> boff, bob, celloff, bkey, bcount, bfill, bbsum;
  DBuf<double> ref, Lp;
  Config cur, plus, minus, next;
  // body-block preconditioner
  int max_blobs = 0;
  DBuf<int> shape_of;
  DBuf<i64> shape_off, shape_offg;
  DBuf<float> shape_B;
  DBuf<double> shape_G;
  // coupled (all-blob) body block for small suspensions
  bool dense_body = false;
  PairMobility pair{};   // blob pair functions of the grid's kernel
  DBuf<float> dM, dP, dE, dB;
  DBuf<double> dN, dNw, dG;
  DBuf<int> dstatus;
  // Newton-Schulz update of dM from the previous configuration's inverse:
  // work matrices, the residual norm, whether dM holds a valid inverse, and
  // how many builds took the warm start
  DBuf<float> dMw, dTw, dUw;
  DBuf<double> dss, dquat;   // dquat: body orientations dM was built at
  bool dM_valid = false, dquat_valid = false;
  long long ns_warm = 0;
  // work vectors (FP64)
  DBuf<double> part, scal, bvec, xvec, xrfd, rres, fnoise, Wst;
  DBuf<double> bodyF, bodyW, bodyWn, blobS;
  double* h_pinned = nullptr;
  int nparts = 0;
  // precision-specific stores
  MGStore<float> mg32;
  KrylovStore<double> kr64;
  KrylovStore<float> kr32;
  DBuf<float> f32a, f32b;
  DBuf<double> small;     // Hessenberg, rotations, g, y, dots
  int total_iters = 0;
  long long reorth_passes = 0, gs_iters = 0;   // host-driven iterations: second passes taken / iterations
  // FGMRES restart cycles captured as CUDA graphs: [precision 0 = FP64, 1 = FP32][with bodies]
  struct CycleGraph {
    cudaGraphExec_t exec = nullptr;
    const void* b = nullptr;
    const void* x = nullptr;
    i64 n = 0;
    long long per_iter = 0, fixed = 0;
  } cgraph[2][2];
  bool use_graphs = true;
  int cap_depth = 0;                       // nesting depth of the conditional body being captured
  cudaStream_t cap_streams[8] = {};         // capture streams, one per nesting depth
  // Device-driven SEM step: the whole step captured as one graph per grid
  // (restart cycles and refinement sweeps in WHILE nodes, the body block's
  // warm-start choice in an IF/ELSE node), run with no host round trip.
  // dstep: seed, step, attempt; dinfo: per solve (rfd, stokes, main) 4 ints
  // (iterations, status, cycles or sweeps, second Gram-Schmidt passes), then
  // [12] rejected, [13] outside flag, [16..19] the refinement's inner solve;
  // drel: per solve relative residual, [3] inner; drst / drsi: refinement
  // state; dwarm: Newton-Schulz builds.
  bool dev = false;
  bool step_graphs = true;      // RBFIB_NO_STEP_GRAPH=1: host-orchestrated steps
  int last_step_dev = 0;        // whether the last SEM step ran as the step graph
  // launch accounting of the step graph: per solve slot the fixed launches of
  // one pass of its WHILE body (a restart cycle, or a refinement sweep with
  // its one-cycle inner solve) and one iteration's launches; the launches
  // outside every WHILE body
  long long cap_body_fixed[3] = {}, cap_per_iter[3] = {}, cap_bodies = 0, cap_outside = 0;
  long long ns_warm_dev = 0;    // Newton-Schulz builds of device-driven steps
  DBuf<unsigned long long> dstep;
  DBuf<int> dinfo, drsi;
  DBuf<double> drel, drst;
  DBuf<long long> dwarm;
  struct StepGraph {
    cudaGraphExec_t exec = nullptr;
    double* q = nullptr;
    double* quat = nullptr;
    rbfib_sem_params p{};
  } sgraph;
  DBuf<int> gst;
  DBuf<double> dpar;
  // kernel timer (roofline reports): events around launches of one class
  int timer_kind = 0;
  std::vector<cudaEvent_t> tev;
  size_t tev_used = 0;
  double timer_bytes = 0.0, timer_flops = 0.0;
  int64_t timer_launches = 0;

  i64 n_total() const { return nfl + 3 * (i64)nbl + 6 * (i64)nb; }
};

namespace {

// Records events around launches of the selected kernel class.
struct TimerScope {
  rbfib_grid* g;
  bool on;
  TimerScope(rbfib_grid* g_, int kind, double bytes, double flops) : g(g_), on(g_->timer_kind == kind) {
    if (!on) return;
    if (g->tev_used + 2 > g->tev.size()) {
      if (g->tev.size() >= 400000) { on = false; return; }
      for (int i = 0; i < 256; ++i) {
        cudaEvent_t e;
        ck(cudaEventCreate(&e));
        g->tev.push_back(e);
      }
    }
    // the stream waits about 25 us first, so the timed launches are queued
    // behind the opening event and it measures them, not host launch gaps
    gpu_delay(50000, g->s);
    ck(cudaEventRecord(g->tev[g->tev_used], g->s));
    g->timer_bytes += bytes;
    g->timer_flops += flops;
    g->timer_launches += 1;
  }
  ~TimerScope() {
    if (on) {
      cudaEventRecord(g->tev[g->tev_used + 1], g->s);
      g->tev_used += 2;
    }
  }
};

enum { TK_MATVEC = 1, TK_SMOOTH = 2, TK_DOT = 3, TK_AXPY = 4, TK_COARSE = 5 };

void drop_graphs(rbfib_grid* g) {
  for (auto& row : g->cgraph)
    for (auto& c : row) {
      if (c.exec) cudaGraphExecDestroy(c.exec);
      c = rbfib_grid::CycleGraph();
    }
  if (g->sgraph.exec) cudaGraphExecDestroy(g->sgraph.exec);
  g->sgraph = rbfib_grid::StepGraph();
}

int fail(rbfib_grid* g, int code, const std::string& msg) {
  if (g) g->err = msg;
  return code;
}

BodyView view_of(rbfib_grid* g, Config& c) {
  BodyView b;
  b.nb = g->nb; b.nbl = g->nbl;
  b.boff = g->boff; b.bob = g->bob; b.perm = c.perm.p;
  b.ref = g->ref; b.q = c.q; b.quat = c.quat; b.r = c.r; b.arm = c.arm;
  b.st64 = c.st64.p; b.st32 = c.st32.p;
  return b;
}

ShapeView shapes_of(rbfib_grid* g) {
  ShapeView v;
  v.max_blobs = g->max_blobs;
  v.shape_of = g->shape_of;
  v.off = g->shape_off;
  v.B = g->shape_B;
  v.offg = g->shape_offg;
  v.G = g->shape_G;
  return v;
}

// --------------------------------------------------------------- multigrid
// Small-array layout inside g->small: [H (m+1)*m | cs m | sn m | g m+1 | y m |
// hcol 128 | hcol2 128 | nrm2 2 | res 2 | bnorm 2]
struct SmallPtrs {
  double *H, *cs, *sn, *gv, *y, *hcol, *hcol2, *nrm2, *res, *bn;
};
SmallPtrs small_ptrs(rbfib_grid* g, int m) {
  SmallPtrs p;
  double* b = g->small;
  p.H = b; b += (size_t)(m + 1) * m;
  p.cs = b; b += m;
  p.sn = b; b += m;
  p.gv = b; b += m + 1;
  p.y = b; b += m;
  p.hcol = b; b += 128;
  p.hcol2 = b; b += 128;
  p.nrm2 = b; b += 2;
  p.res = b; b += 2;
  p.bn = b; b += 2;
  return p;
}

template <typename T>
MGStore<T>& mg_of(rbfib_grid* g);
template <>
MGStore<float>& mg_of<float>(rbfib_grid* g) { return g->mg32; }
template <typename T>
KrylovStore<T>& kr_of(rbfib_grid* g);
template <>
KrylovStore<double>& kr_of<double>(rbfib_grid* g) { return g->kr64; }
template <>
KrylovStore<float>& kr_of<float>(rbfib_grid* g) { return g->kr32; }

// Smoothing sweeps before and after the coarse correction, V(2,2).  V(1,2)
// is marginally faster on the two-sphere grid (one GPU-wide level above the
// coarse solve) but costs 10% more iterations on the 128x128x64 grid (two
// levels); V(2,1) and V(1,1) cost more iterations than they save.
const int kNuPre = 2;
const int kNuPost = 2;
int coarse_sweeps(const Dims& d) { return std::max(d.n[0], std::max(d.n[1], d.n[2])) + 2; }

// Algorithmic FP32 operations of one coarse-level solve by fast
// diagonalisation: per grid six 1D transforms (one FMA per point and
// transform-axis entry) and one division per point.
// Algorithmic bytes of one coarse-level solve: per grid the right-hand
// side read and the solution written (FP32), and its basis table read.
double fd_bytes(const FDParams& P) {
  double b = 0.0;
  for (int g = 0; g < P.ng; ++g)
    b += 4.0 * (2.0 * P.g[g].e[0] * P.g[g].e[1] * P.g[g].e[2] + P.g[g].tabn);
  return b;
}

double fd_flops(const FDParams& P) {
  double f = 0.0;
  for (int g = 0; g < P.ng; ++g) {
    const double n = (double)P.g[g].e[0] * P.g[g].e[1] * P.g[g].e[2];
    f += 2.0 * 2.0 * n * (P.g[g].e[0] + P.g[g].e[1] + P.g[g].e[2]) + n;
  }
  return f;
}

// u0 <- V-cycle approximation of (-eta LL)^{-1} rhs0 (zero initial guess).
// FP32: the levels above the coarse level are smoothed by red-black
// Gauss-Seidel and the coarse level is solved exactly (fast
// diagonalisation); otherwise the coarsest level gets coarse_sweeps sweeps.
template <typename T>
void vcycle_vel(rbfib_grid* g, T* u0, const T* rhs0) {
  MGStore<T>& M = mg_of<T>(g);
  const int L = (int)g->levels.size();
  const T eta = (T)g->desc.eta;
  std::vector<T*> u(L), rhs(L);
  for (int l = 0; l < L; ++l) { u[l] = *M.vu[l]; rhs[l] = *M.vrhs[l]; }
  u[0] = u0;
  rhs[0] = const_cast<T*>(rhs0);
  auto smooth = [&](int l, int color) {
    const Dims& d = g->levels[l].d;
    TimerScope ts(g, l == 0 ? TK_SMOOTH : -1, 2.0 * (double)d.fo[3] * sizeof(T), 4.5 * (double)d.fo[3]);
    vel_rbgs<T>(d, eta, color, u[l], rhs[l], g->s, l == 0 ? g->tune.vrbgs : 256);
  };
  const bool fd = std::is_same<T, float>::value && g->fd_vel >= 0;
  const int lt = fd ? g->fd_vel : L - 1;
  for (int l = 0; l < lt; ++l) {
    const Dims& d = g->levels[l].d;
    // zero guess, then colours 0 and 1 (one launch on uniform spacing)
    bool fused;
    {
      TimerScope ts(g, l == 0 ? TK_SMOOTH : -1, 2.0 * (double)d.fo[3] * sizeof(T), 4.5 * (double)d.fo[3]);
      fused = vel_first2<T>(d, eta, u[l], rhs[l], g->s, l == 0 ? g->tune.vrbgs : 256);
    }
    if (!fused) {
      vel_first<T>(d, eta, u[l], rhs[l], g->s);
      smooth(l, 1);
    }
    for (int s = 1; s < kNuPre; ++s) { smooth(l, 0); smooth(l, 1); }
    vel_restrict_res<T>(d, g->levels[l + 1].d, g->levels[l].cz, eta, u[l], rhs[l], rhs[l + 1], g->s);
  }
  if constexpr (std::is_same<T, float>::value) {
    if (fd) {
      TimerScope ts(g, TK_COARSE, fd_bytes(g->fdv), fd_flops(g->fdv));
      fd_solve(g->fdv, u[lt], rhs[lt], g->fd_tmp, g->s);
    } else {
      vel_coarse<T>(g->levels[L - 1].d, eta, u[L - 1], rhs[L - 1], coarse_sweeps(g->levels[L - 1].d), g->s);
    }
  } else {
    vel_coarse<T>(g->levels[L - 1].d, eta, u[L - 1], rhs[L - 1], coarse_sweeps(g->levels[L - 1].d), g->s);
  }
  for (int l = lt - 1; l >= 0; --l) {
    const Dims& d = g->levels[l].d;
    vel_prolong<T>(d, g->levels[l + 1].d, g->levels[l].cz, u[l + 1], u[l], g->s);
    for (int s = 0; s < kNuPost; ++s) { smooth(l, 1); smooth(l, 0); }
  }
}

// u0 <- V-cycle approximation of (-D G)^{-1} rhs0 (Neumann; rhs0 is scratch)
template <typename T>
void vcycle_p(rbfib_grid* g, T* u0, T* rhs0) {
  MGStore<T>& M = mg_of<T>(g);
  const int L = (int)g->levels.size();
  std::vector<T*> u(L), rhs(L);
  for (int l = 0; l < L; ++l) { u[l] = *M.pu[l]; rhs[l] = *M.prhs[l]; }
  u[0] = u0;
  rhs[0] = rhs0;
  const bool fd = std::is_same<T, float>::value && g->fd_p >= 0;
  const int lt = fd ? g->fd_p : L - 1;
  for (int l = 0; l < lt; ++l) {
    const Dims& d = g->levels[l].d;
    const int bs = l == 0 ? g->tune.prbgs : 256;
    if (!p_first2<T>(d, u[l], rhs[l], g->s, bs)) {   // zero guess, then colours 0 and 1
      p_first<T>(d, u[l], rhs[l], g->s);
      p_rbgs<T>(d, 1, u[l], rhs[l], g->s, bs);
    }
    for (int s = 1; s < kNuPre; ++s) { p_rbgs<T>(d, 0, u[l], rhs[l], g->s, bs); p_rbgs<T>(d, 1, u[l], rhs[l], g->s, bs); }
    p_restrict_res<T>(d, g->levels[l + 1].d, g->levels[l].cz, u[l], rhs[l], rhs[l + 1], g->s);
  }
  if constexpr (std::is_same<T, float>::value) {
    if (fd) {
      TimerScope ts(g, TK_COARSE, fd_bytes(g->fdp), fd_flops(g->fdp));
      fd_solve(g->fdp, u[lt], rhs[lt], g->fd_tmp, g->s);
    } else {
      p_coarse<T>(g->levels[L - 1].d, u[L - 1], rhs[L - 1], coarse_sweeps(g->levels[L - 1].d), g->s);
    }
  } else {
    p_coarse<T>(g->levels[L - 1].d, u[L - 1], rhs[L - 1], coarse_sweeps(g->levels[L - 1].d), g->s);
  }
  for (int l = lt - 1; l >= 0; --l) {
    const Dims& d = g->levels[l].d;
    p_prolong<T>(d, g->levels[l + 1].d, g->levels[l].cz, u[l + 1], u[l], g->s);
    const int bs = l == 0 ? g->tune.prbgs : 256;
    for (int s = 0; s < kNuPost; ++s) { p_rbgs<T>(d, 1, u[l], rhs[l], g->s, bs); p_rbgs<T>(d, 0, u[l], rhs[l], g->s, bs); }
  }
}

// kappa of the pressure block: per axis the walls' share of the viscous drag
// on a flow across it, 12 / H^2 between two no-slip walls, 3 / H^2 (half a
// channel of height 2 H) with one of them free-slip; the smallest of the three
// directions' sums over the two axes across them, so that no wave's drag is
// overstated.  It is that of waves across the narrowest gap, the shortest
// ones: nothing in a slit that is periodic along it, and a small part of what
// waves along a thin channel feel (12 / 96^2 for 12 / 12^2 + 12 / 96^2 in 384 x 96 x
// 12).  Krylov iterations of a fluid-driven and a sphere's solve to 1e-8:
// two-sphere box 33 -> 27 (rigid), channel of 384 x 48 x 12 57 -> 35 (fluid).
double pressure_kappa(const Dims& d) {
  double drag[3];
  for (int b = 0; b < 3; ++b) {
    const double H = d.n[b] * d.h[b];
    const int noslip = d.per[b] ? 0 : (d.gd[2 * b] > 0) + (d.gd[2 * b + 1] > 0);
    drag[b] = noslip == 2 ? 12.0 / (H * H) : (noslip == 1 ? 3.0 / (H * H) : 0.0);
  }
  return std::min(drag[0] + drag[1], std::min(drag[0] + drag[2], drag[1] + drag[2]));
}

// ---------------------------------------------------------- preconditioner
// Block lower-triangular preconditioner of the saddle operator.
// Fluid block (projection method): v~ = (-eta LL)^{-1} r_v (V-cycle),
// q = r_pi + D v~, phi = (-D G)^{-1} q (V-cycle), v = v~ + G phi,
// pi = -eta (q + kappa phi).  -eta q alone (kappa = 0) is exact for periodic
// boxes.  Between no-slip walls a distance H apart a long pressure wave (k H
// small) drives Poiseuille flow instead, for which the pressure operator
// D (-LL)^{-1} G is k^2 H^2 / 12, not 1: kappa = 12 / H^2 adds that limit, as
// the mass term's part does in preconditioners of the unsteady Stokes
// problem (Cahouet and Chabard).  See pressure_kappa.
// Body block: Schur complement [-M K; K^T 0] with M replaced per body by the
// free-space blob mobility of its shape (pair_mobility.cuh), right-hand side
// (r_lam + J v, r_U).
// z64 (optional): the result is also written in FP64 there by the kernels
// that produce each block, which saves a conversion launch.
template <typename T>
void precond(rbfib_grid* g, const T* r, T* z, bool with_bodies, double* z64, double kappa) {
  const Dims& d = g->d;
  T* zv = z;
  MGStore<T>& M = mg_of<T>(g);
  vcycle_vel<T>(g, zv, r);
  T* q = *M.prhs[0];
  T* phi = *M.pu[0];
  div_q<T>(d, zv, r + g->nf, q, g->s);
  vcycle_p<T>(g, phi, q);
  add_grad<T>(d, (T)g->desc.eta, (T)kappa, phi, q, z, z64, g->s);
  if constexpr (std::is_same<T, float>::value) {
    if (with_bodies && g->nb > 0) {
      const BodyView bv = view_of(g, g->cur);
      double* zb64 = z64 ? z64 + g->nfl : nullptr;
      if (g->dense_body) dense_body_apply(g->nbl, g->nb, g->dB, g->dG, r + g->nfl, z + g->nfl, zb64, d, bv.st32, zv, g->s);
      else body_apply(bv, shapes_of(g), r + g->nfl, z + g->nfl, zb64, d, zv, g->s);
    }
  }
}

// The preconditioner always runs in FP32: it only has to approximate A^{-1}
// (FGMRES is flexible), and FP32 halves the bytes of every multigrid sweep and
// avoids GB300's narrow FP64 pipe.  FP64 vectors are converted on the way in;
// on the way out the kernels that finish each block write it in FP64 too.  r32_ready: the Krylov basis kernels already wrote r rounded to
// FP32 into f32a (normalising a new basis vector writes both copies, which
// saves a conversion launch).
void precond_any(rbfib_grid* g, const double* r, double* z, bool with_bodies, bool r32_ready = false) {
  const i64 n = with_bodies ? g->n_total() : g->nfl;
  if (!r32_ready) convert<double, float>(r, g->f32a, n, g->s);
  precond<float>(g, g->f32a, g->f32b, with_bodies, z, g->kappa);
}
void precond_any(rbfib_grid* g, const float* r, float* z, bool with_bodies, bool = false) {
  precond<float>(g, r, z, with_bodies, nullptr, g->kappa);
}
// Where the basis kernels put the FP32 copy of a new FP64 basis vector (the
// FP32 Krylov mode keeps f32a for the right-hand side of its inner solve).
template <typename T> float* basis32(rbfib_grid* g) { return sizeof(T) == 8 ? g->f32a.p : nullptr; }

// y = A x (saddle operator; fluid-only when with_bodies is false)
template <typename T>
void apply_A(rbfib_grid* g, const T* x, T* y, bool with_bodies) {
  const double nbytes = 2.0 * (double)(with_bodies ? g->n_total() : g->nfl) * sizeof(T) +
                        (with_bodies ? 24.0 * g->nbl + 56.0 * g->nb : 0.0);
  // operations: 10 per momentum row, 6 per divergence row, about 400 per blob
  // (interpolation and spreading, 3 x 27 weighted terms each, and K, K^T)
  const double nflops = 10.0 * g->nf + 6.0 * g->nc + (with_bodies ? 400.0 * g->nbl : 0.0);
  TimerScope ts(g, TK_MATVEC, nbytes, nflops);
  const int sbs = sizeof(T) == 8 ? g->tune.stokes64 : g->tune.stokes32;
  stokes_apply<T>(g->d, (T)g->desc.eta, x, x + g->nf, y, y + g->nf, g->s, sbs > 0 ? sbs : 256);
  if (with_bodies && g->nb > 0) {
    const T* xl = x + g->nfl;
    const T* xU = xl + 3 * (i64)g->nbl;
    saddle_bodies<T>(g->d, view_of(g, g->cur), x, xl, xU, y, y + g->nfl, y + g->nfl + 3 * (i64)g->nbl, g->s);
  }
}

// Selective re-orthogonalisation threshold tau^2 (ReorthCtl): the second
// Gram-Schmidt pass runs when the first keeps less than a fraction tau of
// ||w||.  FP64: tau = 1e-3, so a skipped pass leaves at most about
// 1e3 eps = 2e-13 of lost orthogonality per basis vector, far below what a
// solve to 1e-8 (or the tests' 1e-12) can notice, and the true residual
// checked at the end of every restart cycle guards the result; on the
// two-sphere solves the first pass keeps well above that, so the FP64 sweeps
// halve.  FP32 (the refinement's inner solves to 1e-4, where eps is 6e-8):
// tau = 1e-2 (at most about 6e-6 lost per vector); the DGKS constant
// 1/sqrt(2) re-orthogonalised nearly always and made the refined two-sphere
// step 10% slower (68.7 against 76.5 steps/s) with the same iterations.
// RBFIB_REORTH_TAU64 and RBFIB_REORTH_TAU32 override the values (1
// re-orthogonalises always).
double reorth_tau2(bool fp64) {
  static const double t64 = [] {
    const char* e = std::getenv("RBFIB_REORTH_TAU64");
    const double t = e ? std::atof(e) : 1e-3;
    return t * t;
  }();
  static const double t32 = [] {
    const char* e = std::getenv("RBFIB_REORTH_TAU32");
    const double t = e ? std::atof(e) : 1e-2;
    return t * t;
  }();
  return fp64 ? t64 : t32;
}

int read_int(rbfib_grid* g, const int* dev) {
  int* hi = (int*)(g->h_pinned + 44);
  ck(cudaMemcpyAsync(hi, dev, sizeof(int), cudaMemcpyDeviceToHost, g->s));
  ck(cudaStreamSynchronize(g->s));
  return hi[0];
}

double read_scalar(rbfib_grid* g, const double* dev) {
  ck(cudaMemcpyAsync(g->h_pinned, dev, sizeof(double), cudaMemcpyDeviceToHost, g->s));
  ck(cudaStreamSynchronize(g->s));
  return g->h_pinned[0];
}

// Right-preconditioned flexible GMRES(m) with classical Gram-Schmidt and one
// re-orthogonalisation, inner products weighted by dV on the fluid unknowns.
// Solves A x = b from x = 0 to ||b - A x||_W <= rtol ||b||_W.
// Returns 0, RBFIB_ENOCONV or RBFIB_ENAN; iters and relres report progress.
template <typename T>
int fgmres(rbfib_grid* g, const T* b, T* x, bool with_bodies, double rtol, int maxit, int& iters, double& relres) {
  KrylovStore<T>& K = kr_of<T>(g);
  const int m = K.m;
  const i64 n = with_bodies ? g->n_total() : g->nfl;
  const i64 ld = K.n;
  const i64 nfl = g->nfl;
  const double wf = g->dV;
  SmallPtrs sp = small_ptrs(g, m);
  T* V = K.V;
  T* Z = K.Z;
  T* w = K.w;
  iters = 0;
  relres = 0.0;
  multi_dot<T>(b, b, ld, 1, n, nfl, wf, g->part, g->nparts, sp.bn, g->s);
  const double bnorm = std::sqrt(std::max(read_scalar(g, sp.bn), 0.0));
  ck(cudaMemsetAsync(x, 0, sizeof(T) * n, g->s));
  if (!(bnorm > 0.0)) {
    if (std::isnan(bnorm)) return RBFIB_ENAN;
    return 0;
  }
  // r = b (x = 0)
  ck(cudaMemcpyAsync(w, b, sizeof(T) * n, cudaMemcpyDeviceToDevice, g->s));
  double beta = bnorm;
  for (;;) {
    // V_0 = r / beta ; g = (beta, 0, ...)
    ck(cudaMemsetAsync(sp.gv, 0, sizeof(double) * (m + 1), g->s));
    g->h_pinned[1] = beta;
    ck(cudaMemcpyAsync(sp.gv, g->h_pinned + 1, sizeof(double), cudaMemcpyHostToDevice, g->s));
    scale_by<T>(V, w, sp.gv, 1, n, g->s, basis32<T>(g));
    int k = 0;
    for (int j = 0; j < m; ++j) {
      T* vj = V + (i64)j * ld;
      T* zj = Z + (i64)j * ld;
      precond_any(g, vj, zj, with_bodies, true);
      apply_A<T>(g, zj, w, with_bodies);
      const double bd = (double)(j + 2) * n * sizeof(T), ba = (double)(j + 3) * n * sizeof(T);
      const double fd = 2.0 * (j + 1) * n, fa = 2.0 * (j + 2) * n;
      const ReorthCtl rc{g->gst.p + 4, sp.hcol2, reorth_tau2(sizeof(T) == 8), 0, 0};
      { TimerScope ts(g, TK_DOT, bd, fd); multi_dot<T>(w, V, ld, j + 1, n, nfl, wf, g->part, g->nparts, sp.hcol, g->s); }
      { TimerScope ts(g, TK_AXPY, ba, fa); multi_axpy<T>(w, V, ld, j + 1, sp.hcol, -1.0, n, nfl, wf, g->part, g->nparts, sp.nrm2, g->s, &rc); }
      // host-driven iterations read the decision, so that the kernel timer
      // only counts second passes that run
      if (read_int(g, g->gst.p + 4)) {
        ++g->reorth_passes;
        { TimerScope ts(g, TK_DOT, bd, fd); multi_dot<T>(w, V, ld, j + 1, n, nfl, wf, g->part, g->nparts, sp.hcol2, g->s); }
        { TimerScope ts(g, TK_AXPY, ba, fa); multi_axpy<T>(w, V, ld, j + 1, sp.hcol2, -1.0, n, nfl, wf, g->part, g->nparts, sp.nrm2, g->s); }
      }
      ++g->gs_iters;
      givens_step(sp.H, m + 1, sp.cs, sp.sn, sp.gv, j, sp.hcol, sp.hcol2, sp.nrm2, sp.res, g->s);
      scale_by<T>(V + (i64)(j + 1) * ld, w, sp.nrm2, 2, n, g->s, basis32<T>(g));
      ++iters;
      k = j + 1;
      const double res = read_scalar(g, sp.res);
      if (std::isnan(res)) return RBFIB_ENAN;
      if (res <= rtol * bnorm || iters >= maxit) break;
    }
    tri_solve(sp.H, m + 1, sp.gv, k, sp.y, g->s);
    multi_axpy<T>(x, Z, ld, k, sp.y, 1.0, n, nfl, wf, g->part, g->nparts, nullptr, g->s);
    // true residual
    apply_A<T>(g, x, w, with_bodies);
    axpby<T>(w, b, 1.0, -1.0, n, g->s);   // w = b - A x
    multi_dot<T>(w, w, ld, 1, n, nfl, wf, g->part, g->nparts, sp.bn, g->s);
    beta = std::sqrt(std::max(read_scalar(g, sp.bn), 0.0));
    relres = beta / bnorm;
    if (std::isnan(relres)) return RBFIB_ENAN;
    if (relres <= rtol) return 0;
    if (iters >= maxit) return RBFIB_ENOCONV;
  }
}

// ------------------------------------------------------- graph capture
// Conditional nodes are added to the graph being captured on g->s; each body
// graph is captured on a stream of a small pool indexed by nesting depth
// (a cycle graph nests the reorthogonalisation IF inside the iteration IF;
// the device-driven SEM step puts cycles inside WHILE nodes, and the
// refinement's inner solve inside another WHILE).
constexpr int kCapDepth = 8;

cudaStream_t cap_stream(rbfib_grid* g, int depth) {
  if (depth >= kCapDepth) throw CudaError{cudaErrorInvalidValue};
  if (!g->cap_streams[depth]) ck(cudaStreamCreateWithFlags(&g->cap_streams[depth], cudaStreamNonBlocking));
  return g->cap_streams[depth];
}

cudaGraphConditionalHandle new_handle(rbfib_grid* g, unsigned dflt) {
  cudaStreamCaptureStatus cst;
  cudaGraph_t capg = nullptr;
  ck(cudaStreamGetCaptureInfo(g->s, &cst, nullptr, &capg, nullptr, nullptr, nullptr));
  cudaGraphConditionalHandle h;
  ck(cudaGraphConditionalHandleCreate(&h, capg, dflt, cudaGraphCondAssignDefault));
  return h;
}

// Adds a conditional node (IF with one or two bodies, or WHILE) after the
// work captured so far on g->s and captures body b with fill(b).
template <typename F>
void cond_node(rbfib_grid* g, cudaGraphConditionalHandle h, cudaGraphConditionalNodeType type, int nbody, F fill) {
  cudaStreamCaptureStatus cst;
  cudaGraph_t capg = nullptr;
  const cudaGraphNode_t* deps = nullptr;
  size_t nd = 0;
  ck(cudaStreamGetCaptureInfo(g->s, &cst, nullptr, &capg, &deps, nullptr, &nd));
  cudaGraphNodeParams p = {};
  p.type = cudaGraphNodeTypeConditional;
  p.conditional.handle = h;
  p.conditional.type = type;
  p.conditional.size = nbody;
  cudaGraphNode_t node;
  ck(cudaGraphAddNode(&node, capg, deps, nullptr, nd, &p));
  ck(cudaStreamUpdateCaptureDependencies(g->s, &node, nullptr, 1, cudaStreamSetCaptureDependencies));
  cudaStream_t outer = g->s;
  const int depth = ++g->cap_depth;
  for (int bi = 0; bi < nbody; ++bi) {
    cudaGraph_t body = p.conditional.phGraph_out[bi];
    cudaStream_t sb = cap_stream(g, depth);
    ck(cudaStreamBeginCaptureToGraph(sb, body, nullptr, nullptr, 0, cudaStreamCaptureModeRelaxed));
    g->s = sb;
    try {
      fill(bi);
    } catch (...) {
      cudaGraph_t t;
      cudaStreamEndCapture(sb, &t);
      g->s = outer;
      --g->cap_depth;
      throw;
    }
    ck(cudaStreamEndCapture(sb, &body));
    g->s = outer;
  }
  --g->cap_depth;
}

// One iteration of a captured restart cycle (the body of its loop).  The
// column j = ist[0] is read on the device: the preconditioner takes its input
// from a fixed FP32 copy of the newest basis vector and leaves its result in
// a fixed vector, and only the sweeps and the last launch look j up.  The
// second Gram-Schmidt pass sits in a nested IF node whose condition the
// first pass's multi-axpy sets (ReorthCtl).
template <typename T>
void capture_iteration(rbfib_grid* g, bool wb, cudaGraphConditionalHandle loop) {
  KrylovStore<T>& K = kr_of<T>(g);
  const int m = K.m;
  const i64 n = wb ? g->n_total() : g->nfl, ld = K.n, nfl = g->nfl;
  const double wf = g->dV;
  SmallPtrs sp = small_ptrs(g, m);
  T* V = K.V;
  T* w = K.w;
  int* kdev = g->gst;
  if constexpr (sizeof(T) == 8) precond<float>(g, K.v32, g->f32b, wb, K.z, g->kappa);
  else precond<float>(g, K.v32, K.z, wb, nullptr, g->kappa);
  apply_A<T>(g, K.z, w, wb);
  const cudaGraphConditionalHandle h2 = new_handle(g, 0u);
  const ReorthCtl rc{g->gst.p + 4, sp.hcol2, reorth_tau2(sizeof(T) == 8), h2, 1};
  multi_dot<T>(w, V, ld, m, n, nfl, wf, g->part, g->nparts, sp.hcol, g->s, kdev);
  multi_axpy<T>(w, V, ld, m, sp.hcol, -1.0, n, nfl, wf, g->part, g->nparts, sp.nrm2, g->s, &rc, kdev);
  cond_node(g, h2, cudaGraphCondTypeIf, 1, [&](int) {
    multi_dot<T>(w, V, ld, m, n, nfl, wf, g->part, g->nparts, sp.hcol2, g->s, kdev);
    multi_axpy<T>(w, V, ld, m, sp.hcol2, -1.0, n, nfl, wf, g->part, g->nparts, sp.nrm2, g->s, nullptr, kdev);
  });
  scale_givens<T>(V, K.Z, ld, w, K.z, n, K.v32, sp.H, m, sp.cs, sp.sn, sp.gv, sp.hcol, sp.hcol2, sp.nrm2, sp.res, g->gst,
                  g->dpar, loop, g->s);
}

// One restart cycle of FGMRES(m), captured on g->s: the cycle start, the
// Arnoldi iterations in a WHILE node whose condition each iteration's Givens
// update sets (converged, budget, m columns), then the solution update and the
// true residual w = b - A x with its norm in dpar[2].  The loop holds one
// iteration's nodes where a chain of m IF nodes held m: skipped nodes cost
// 1.5-2 us each, and capture and instantiation m times as many.  per_iter (if
// not null) receives the launches of one iteration with its gated second pass
// (two launches).
template <typename T>
void capture_cycle(rbfib_grid* g, const T* b, T* x, bool wb, long long* per_iter) {
  KrylovStore<T>& K = kr_of<T>(g);
  const int m = K.m;
  const i64 n = wb ? g->n_total() : g->nfl, ld = K.n, nfl = g->nfl;
  const double wf = g->dV;
  SmallPtrs sp = small_ptrs(g, m);
  const cudaGraphConditionalHandle loop = new_handle(g, 1u);
  fg_start<T>(K.V, K.w, n, sp.gv, m, g->gst, g->dpar, g->s, K.v32, loop);
  const long long a0 = rbfib::g_launches.load();
  cond_node(g, loop, cudaGraphCondTypeWhile, 1, [&](int) { capture_iteration<T>(g, wb, loop); });
  if (per_iter) *per_iter = (long long)rbfib::g_launches.load() - a0;
  tri_solve_dev(sp.H, m + 1, sp.gv, g->gst, sp.y, g->s);
  multi_axpy_dev<T>(x, K.Z, ld, g->gst, sp.y, 1.0, n, g->nparts, g->s);
  apply_A<T>(g, x, K.w, wb);
  axpby<T>(K.w, b, 1.0, -1.0, n, g->s);
  multi_dot<T>(K.w, K.w, ld, 1, n, nfl, wf, g->part, g->nparts, g->dpar + 2, g->s);
}

// A restart cycle as a graph of its own (the host-orchestrated solves launch
// one per restart and read three numbers).
template <typename T>
bool build_cycle_graph(rbfib_grid* g, const T* b, T* x, bool wb, rbfib_grid::CycleGraph& G) {
  const i64 n = wb ? g->n_total() : g->nfl;
  cudaStream_t s0 = g->s, sc = nullptr;
  const int saved_timer = g->timer_kind;
  bool ok = true;
  const long long l0 = rbfib::g_launches.load();
  long long per_iter = 0;
  cudaGraph_t graph = nullptr;
  if (cudaStreamCreateWithFlags(&sc, cudaStreamNonBlocking) != cudaSuccess) return false;
  g->timer_kind = 0;
  g->s = sc;
  g->cap_depth = 0;
  try {
    ck(cudaStreamBeginCapture(sc, cudaStreamCaptureModeRelaxed));
    capture_cycle<T>(g, b, x, wb, &per_iter);
    ck(cudaStreamEndCapture(sc, &graph));
    ck(cudaGraphInstantiate(&G.exec, graph, 0));
  } catch (CudaError&) {
    ok = false;
    cudaStreamCaptureStatus cst;
    if (cudaStreamIsCapturing(sc, &cst) == cudaSuccess && cst != cudaStreamCaptureStatusNone) {
      cudaGraph_t t = nullptr;
      cudaStreamEndCapture(sc, &t);
      if (t) cudaGraphDestroy(t);
    }
    cudaGetLastError();
  }
  if (graph) cudaGraphDestroy(graph);
  g->s = s0;
  g->timer_kind = saved_timer;
  g->cap_depth = 0;
  cudaStreamDestroy(sc);
  const long long captured = (long long)rbfib::g_launches.load() - l0;
  rbfib::g_launches.fetch_sub((unsigned long long)captured);   // captured, not launched
  // an iteration's launches, counting its gated second pass (two launches)
  G.per_iter = per_iter;
  G.fixed = captured - G.per_iter;
  G.b = b; G.x = x; G.n = n;
  return ok;
}

template <typename T>
int fgmres_graph(rbfib_grid* g, const T* b, T* x, bool wb, double rtol, int maxit, int& iters, double& relres) {
  KrylovStore<T>& K = kr_of<T>(g);
  const i64 n = wb ? g->n_total() : g->nfl, ld = K.n, nfl = g->nfl;
  const double wf = g->dV;
  SmallPtrs sp = small_ptrs(g, K.m);
  rbfib_grid::CycleGraph& G = g->cgraph[sizeof(T) == 8 ? 0 : 1][wb ? 1 : 0];
  if (G.exec && (G.b != b || G.x != x || G.n != n)) { cudaGraphExecDestroy(G.exec); G = rbfib_grid::CycleGraph(); }
  if (!G.exec && !build_cycle_graph<T>(g, b, x, wb, G)) {
    g->use_graphs = false;
    return fgmres<T>(g, b, x, wb, rtol, maxit, iters, relres);
  }
  iters = 0;
  relres = 0.0;
  multi_dot<T>(b, b, ld, 1, n, nfl, wf, g->part, g->nparts, sp.bn, g->s);
  const double bnorm = std::sqrt(std::max(read_scalar(g, sp.bn), 0.0));
  ck(cudaMemsetAsync(x, 0, sizeof(T) * n, g->s));
  if (!(bnorm > 0.0)) return std::isnan(bnorm) ? RBFIB_ENAN : 0;
  double* hp = g->h_pinned + 8;
  hp[0] = rtol * bnorm;
  hp[1] = (double)maxit;
  hp[2] = bnorm * bnorm;
  ck(cudaMemcpyAsync(g->dpar, hp, sizeof(double) * 3, cudaMemcpyHostToDevice, g->s));
  ck(cudaMemsetAsync(g->gst, 0, sizeof(int) * 8, g->s));
  ck(cudaMemcpyAsync(K.w, b, sizeof(T) * n, cudaMemcpyDeviceToDevice, g->s));
  int* hi = (int*)(g->h_pinned + 16);
  int passes = 0;
  for (;;) {
    ck(cudaGraphLaunch(G.exec, g->s));
    ck(cudaMemcpyAsync(hi, g->gst, sizeof(int) * 8, cudaMemcpyDeviceToHost, g->s));
    ck(cudaMemcpyAsync(hp + 3, g->dpar + 2, sizeof(double), cudaMemcpyDeviceToHost, g->s));
    ck(cudaStreamSynchronize(g->s));
    const int k = hi[0];
    // launches that ran: the fixed part, k iterations without their gated
    // second Gram-Schmidt pass (two launches), and the second passes taken
    const long long taken = hi[5] - passes;
    passes = hi[5];
    g->reorth_passes += taken;
    g->gs_iters += k;
    rbfib::g_launches.fetch_add((unsigned long long)(G.fixed + (long long)k * (G.per_iter - 2) + 2 * taken));
    iters = hi[1];
    relres = std::sqrt(std::max(hp[3], 0.0)) / bnorm;
    if (std::isnan(relres)) return RBFIB_ENAN;
    if (relres <= rtol) return 0;
    if (iters >= maxit || k == 0) return RBFIB_ENOCONV;
  }
}

// --------------------------------------------------------------- set-up
void build_levels(rbfib_grid* g) {
  g->levels.clear();
  Level L0;
  double h3[3] = {g->desc.h, g->desc.h, g->desc.h};
  L0.d = make_dims(g->desc.n, g->desc.periodic, h3);
  set_free_slip(L0.d, g->desc.free_slip);
  g->levels.push_back(L0);
  for (;;) {
    Level& cur = g->levels.back();
    int cz[3];
    int any = 0;
    for (int a = 0; a < 3; ++a) {
      cz[a] = (cur.d.n[a] % 2 == 0 && cur.d.n[a] >= 4) ? 1 : 0;
      any |= cz[a];
    }
    if (!any || cur.d.nc <= 64) { cur.cz = make_int3(0, 0, 0); break; }
    cur.cz = make_int3(cz[0], cz[1], cz[2]);
    int n2[3], per[3];
    double h2[3];
    for (int a = 0; a < 3; ++a) {
      n2[a] = cz[a] ? cur.d.n[a] / 2 : cur.d.n[a];
      h2[a] = cz[a] ? 2.0 * cur.d.h[a] : cur.d.h[a];
      per[a] = cur.d.per[a];
    }
    Level nx;
    nx.d = make_dims(n2, per, h2);
    for (int w = 0; w < 6; ++w) nx.d.gd[w] = cur.d.gd[w];
    g->levels.push_back(nx);
  }
}

// Coarse levels of the FP32 V-cycles: the finest level whose grids all fit
// the exact solve (usually the grid itself), for the velocity components and
// for the pressure.
void build_fd(rbfib_grid* g) {
  std::vector<float> tab;
  g->fd_vel = g->fd_p = -1;
  std::string why;
  for (int l = 0; l < (int)g->levels.size() && g->fd_vel < 0; ++l)
    if (fd_plan(g->levels[l].d, true, g->desc.eta, tab, g->fdv, why)) g->fd_vel = l;
  for (int l = 0; l < (int)g->levels.size() && g->fd_p < 0; ++l)
    if (fd_plan(g->levels[l].d, false, 1.0, tab, g->fdp, why)) g->fd_p = l;
  if (tab.empty()) return;
  {
    // coefficients of the wide solve: as many floats as the larger level array
    i64 m = 0;
    if (g->fd_vel >= 0) m = std::max(m, g->levels[g->fd_vel].d.fo[3]);
    if (g->fd_p >= 0) m = std::max(m, g->levels[g->fd_p].d.nc);
    g->fd_tmp.alloc((size_t)std::max<i64>(m, 1));
  }
  g->fd_tab.alloc(tab.size());
  ck(cudaMemcpyAsync(g->fd_tab.p, tab.data(), sizeof(float) * tab.size(), cudaMemcpyHostToDevice, g->s));
  ck(cudaStreamSynchronize(g->s));
  g->fdv.tab = g->fd_tab.p;
  g->fdp.tab = g->fd_tab.p;
}

void build_stress_layout(rbfib_grid* g) {
  i64 off = 0;
  for (int a = 0; a < 3; ++a) {
    for (int bb = 0; bb < 3; ++bb) {
      int b = (bb == 0) ? a : (bb == 1 ? (a == 0 ? 1 : 0) : (a == 2 ? 1 : 2));
      int* e = g->stress.ext[a][b];
      for (int ax = 0; ax < 3; ++ax) e[ax] = g->d.n[ax];
      if (b != a) {
        e[a] = g->d.fe[a][a];
        e[b] = g->d.per[b] ? g->d.n[b] : g->d.n[b] + 1;
      }
      g->stress.off[a][b] = off;
      off += (i64)e[0] * e[1] * e[2];
    }
  }
  g->stress.total = off;
}

// dense symmetric positive definite inverse (Cholesky), n small
bool spd_inverse(std::vector<double>& A, int n) {
  std::vector<double> L(A);
  for (int j = 0; j < n; ++j) {
    double s = L[(size_t)j * n + j];
    for (int k = 0; k < j; ++k) s -= L[(size_t)j * n + k] * L[(size_t)j * n + k];
    if (!(s > 0.0)) return false;
    const double d = std::sqrt(s);
    L[(size_t)j * n + j] = d;
    for (int i = j + 1; i < n; ++i) {
      double t = L[(size_t)i * n + j];
      for (int k = 0; k < j; ++k) t -= L[(size_t)i * n + k] * L[(size_t)j * n + k];
      L[(size_t)i * n + j] = t / d;
    }
  }
  // inverse column by column
  std::vector<double> inv((size_t)n * n), y(n);
  for (int c = 0; c < n; ++c) {
    for (int i = 0; i < n; ++i) {
      double t = (i == c) ? 1.0 : 0.0;
      for (int k = 0; k < i; ++k) t -= L[(size_t)i * n + k] * y[k];
      y[i] = t / L[(size_t)i * n + i];
    }
    for (int i = n - 1; i >= 0; --i) {
      double t = y[i];
      for (int k = i + 1; k < n; ++k) t -= L[(size_t)k * n + i] * inv[(size_t)k * n + c];
      inv[(size_t)i * n + c] = t / L[(size_t)i * n + i];
    }
  }
  A.swap(inv);
  return true;
}

// free-space mobility of blobs x (n x 3) (pair_mobility.cuh), its diagonal
// raised up times as much; false if two blobs share one place
bool pair_matrix(const double* x, int nbp, const PairMobility& P, double h, double eta, double up,
                 std::vector<double>& M) {
  const int n3 = 3 * nbp;
  M.assign((size_t)n3 * n3, 0.0);
  for (int i = 0; i < nbp; ++i) {
    int near = 0;
    for (int pass = 0; pass < 2; ++pass)   // neighbours counted, then the blocks
      for (int j = 0; j < nbp; ++j) {
        const double d[3] = {(x[3 * i] - x[3 * j]) / h, (x[3 * i + 1] - x[3 * j + 1]) / h, (x[3 * i + 2] - x[3 * j + 2]) / h};
        if (pass == 0) {
          near += d[0] * d[0] + d[1] * d[1] + d[2] * d[2] < kPairNear * kPairNear;
          continue;
        }
        double B[9];
        pair_block(P, d, i == j ? up * pair_raise(P, near) : 0.0, B);
        if (std::isnan(B[0])) return false;
        for (int p = 0; p < 3; ++p)
          for (int q = 0; q < 3; ++q) M[(size_t)(3 * i + p) * n3 + 3 * j + q] = B[3 * p + q] / (eta * h);
      }
  }
  return true;
}

// Its inverse.  The pair functions are positive definite, so the diagonal as
// it stands suffices for every body tried (pair_raise); should rounding leave
// one that it does not, the diagonal grows until there is a factor, since this
// matrix only preconditions: distinct blobs are never refused.
bool pair_inverse(const double* x, int nbp, const PairMobility& P, double h, double eta, std::vector<double>& M) {
  for (double up = 1.0; up < 1e8; up *= 4.0) {
    if (!pair_matrix(x, nbp, P, h, eta, up, M)) return false;
    if (spd_inverse(M, 3 * nbp)) return true;
  }
  return false;
}

bool inverse6(double A[36]) {
  double aug[6][12];
  for (int i = 0; i < 6; ++i)
    for (int j = 0; j < 12; ++j) aug[i][j] = j < 6 ? A[6 * i + j] : (j - 6 == i ? 1.0 : 0.0);
  for (int c = 0; c < 6; ++c) {
    int piv = c;
    for (int r = c + 1; r < 6; ++r)
      if (std::fabs(aug[r][c]) > std::fabs(aug[piv][c])) piv = r;
    if (aug[piv][c] == 0.0) return false;
    for (int j = 0; j < 12; ++j) std::swap(aug[c][j], aug[piv][j]);
    const double d = aug[c][c];
    for (int j = 0; j < 12; ++j) aug[c][j] /= d;
    for (int r = 0; r < 6; ++r) {
      if (r == c) continue;
      const double f = aug[r][c];
      for (int j = 0; j < 12; ++j) aug[r][j] -= f * aug[c][j];
    }
  }
  for (int i = 0; i < 6; ++i)
    for (int j = 0; j < 6; ++j) A[6 * i + j] = aug[i][j + 6];
  return true;
}

// Coupled body block for the blob positions r (arms arm) of bodies with
// orientations quat (NULL: not known, as after rbfib_set_blob_positions):
// warm-started from the current inverse when there is one
// (dense_body_build).
// A zero pivot in either Gauss-Jordan inversion (the FP32 blob block or the
// FP64 body block) leaves the block invalid and fails the calling entry
// point with RBFIB_EINTERNAL.
void build_body_block(rbfib_grid* g, const double* r, const double* arm, const double* quat) {
  const double* qold = (quat && g->dquat_valid) ? g->dquat.p : nullptr;
  if (g->dev) {
    // captured: the warm start (the step graph is built only when the block
    // holds a valid inverse) with the choice between Newton-Schulz and
    // Gauss-Jordan made on the device; the status goes to dinfo[13]
    ck(cudaMemsetAsync(g->dstatus, 0, sizeof(int), g->s));
    dense_body_mobility(g->nbl, r, g->pair, g->desc.h, g->desc.eta, g->dMw, g->s);
    if (dense_body_warm(g->nbl)) {
      dense_body_warm_start(g->nbl, g->bob, quat, qold, g->dM, g->dMw, g->dTw, g->dss, g->s);
      const cudaGraphConditionalHandle h = new_handle(g, 0u);
      ns_decide(g->dss, h, g->dwarm, g->s);
      cond_node(g, h, cudaGraphCondTypeIf, 2, [&](int branch) {
        if (branch == 0) dense_body_ns(g->nbl, g->dM, g->dMw, g->dTw, g->dUw, g->dss, g->s);
        else dense_body_gj(g->nbl, g->dM, g->dMw, g->dUw, g->dstatus, g->s);
      });
    } else {
      dense_body_gj(g->nbl, g->dM, g->dMw, g->dUw, g->dstatus, g->s);
    }
    dense_body_finish(g->nbl, g->nb, g->boff, arm, g->dM, g->dP, g->dN, g->dNw, g->dstatus, g->s);
    dense_body_matrix(g->nbl, g->nb, g->dM, g->dP, g->dN, g->dE, g->dB, g->dG, g->s);
    ck(cudaMemcpyAsync(g->dinfo.p + 13, g->dstatus.p, sizeof(int), cudaMemcpyDeviceToDevice, g->s));
    if (quat) ck(cudaMemcpyAsync(g->dquat.p, quat, sizeof(double) * 4 * g->nb, cudaMemcpyDeviceToDevice, g->s));
    return;
  }
  bool used = false;
  const bool warm = g->dM_valid;
  g->dM_valid = false;
  ck(dense_body_build(g->nbl, g->nb, g->boff, g->bob, r, arm, quat, qold, g->pair, g->desc.h, g->desc.eta, g->dM, g->dP,
                      g->dN, g->dstatus, g->dMw, g->dTw, g->dUw, g->dNw, g->dss, g->h_pinned + 40, warm, g->s, &used));
  dense_body_matrix(g->nbl, g->nb, g->dM, g->dP, g->dN, g->dE, g->dB, g->dG, g->s);
  int* hstat = (int*)(g->h_pinned + 42);
  ck(cudaMemcpyAsync(hstat, g->dstatus, sizeof(int), cudaMemcpyDeviceToHost, g->s));
  ck(cudaStreamSynchronize(g->s));
  if (*hstat != 0) {
    g->dquat_valid = false;
    CudaError err{cudaSuccess};
    err.code = RBFIB_EINTERNAL;
    err.msg = "body block: zero pivot in the Gauss-Jordan inversion";
    throw err;
  }
  g->dM_valid = true;
  g->dquat_valid = quat != nullptr;
  if (quat) ck(cudaMemcpyAsync(g->dquat.p, quat, sizeof(double) * 4 * g->nb, cudaMemcpyDeviceToDevice, g->s));
  if (used) ++g->ns_warm;
}

void refresh_config(rbfib_grid* g, Config& c, bool bin) {
  geometry(g->nbl, g->bob, g->ref, c.q, c.quat, c.r, c.arm, g->s);
  if (bin) {
    binning(g->d, g->nbl, c.r, c.perm, g->celloff, g->bkey, g->bcount, g->bfill, g->bbsum, g->s);
    stencil_build(g->d, g->nbl, c.r, c.st64, c.st32, g->s);
    if (g->dense_body) build_body_block(g, c.r, c.arm, c.quat);
  }
}

void alloc_config(rbfib_grid* g, Config& c) {
  c.q.alloc(3 * (size_t)g->nb);
  c.quat.alloc(4 * (size_t)g->nb);
  c.r.alloc(3 * (size_t)g->nbl);
  c.arm.alloc(3 * (size_t)g->nbl);
  c.perm.alloc((size_t)g->nbl);
  c.st64.alloc(3 * (size_t)g->nbl);
  c.st32.alloc(3 * (size_t)g->nbl);
}

void alloc_solver(rbfib_grid* g) {
  const i64 n = g->n_total();
  const int m = g->desc.restart;
  if (g->desc.precision == RBFIB_FP64) {
    if (g->kr64.n < n || g->kr64.m != m) g->kr64.build(m, n);
  } else {
    if (g->kr32.n < n || g->kr32.m != m) g->kr32.build(m, n);
    g->rres.ensure(n);
  }
  g->f32a.ensure(n);
  g->f32b.ensure(n);
  g->bvec.ensure(n); g->xvec.ensure(n); g->xrfd.ensure(n);
}

// Appends the body-block matrix of a shape of n blobs x (body frame; k_body.cu),
// its rows of lambda to sB and of U to sG.  Returns why there is none, or null.
const char* shape_matrix(const rbfib_grid* g, const double* x, int n, std::vector<float>& sB, std::vector<double>& sG) {
  const int n3 = 3 * n, ld = body_ld(n3 + 6);
  std::vector<double> M;
  if (!pair_inverse(x, n, g->pair, g->desc.h, g->desc.eta, M)) return "blob mobility of a shape is singular";
  std::vector<double> K((size_t)n3 * 6, 0.0), P((size_t)n3 * 6, 0.0), E((size_t)n3 * 6, 0.0);
  for (int i = 0; i < n; ++i) {
    const double* r = x + 3 * i;
    for (int a = 0; a < 3; ++a) K[(size_t)(3 * i + a) * 6 + a] = 1.0;
    // w x r = -[r]_x w
    K[(size_t)(3 * i + 0) * 6 + 4] = r[2];  K[(size_t)(3 * i + 0) * 6 + 5] = -r[1];
    K[(size_t)(3 * i + 1) * 6 + 3] = -r[2]; K[(size_t)(3 * i + 1) * 6 + 5] = r[0];
    K[(size_t)(3 * i + 2) * 6 + 3] = r[1];  K[(size_t)(3 * i + 2) * 6 + 4] = -r[0];
  }
  double N[36] = {0};
  for (int r = 0; r < n3; ++r)
    for (int k = 0; k < n3; ++k)
      for (int c = 0; c < 6; ++c) P[(size_t)r * 6 + c] += M[(size_t)r * n3 + k] * K[(size_t)k * 6 + c];
  for (int k = 0; k < n3; ++k)
    for (int r = 0; r < 6; ++r)
      for (int c = 0; c < 6; ++c) N[6 * r + c] += K[(size_t)k * 6 + r] * P[(size_t)k * 6 + c];
  if (!inverse6(N)) return "body resistance is singular";
  for (int r = 0; r < n3; ++r)
    for (int c = 0; c < 6; ++c)
      for (int k = 0; k < 6; ++k) E[(size_t)r * 6 + c] += P[(size_t)r * 6 + k] * N[6 * k + c];
  for (int r = 0; r < n3; ++r)
    for (int c = 0; c < ld; ++c) {
      double v = 0.0;
      if (c < n3) {
        v = -M[(size_t)r * n3 + c];
        for (int k = 0; k < 6; ++k) v += E[(size_t)r * 6 + k] * P[(size_t)c * 6 + k];
      } else if (c < n3 + 6) {
        v = E[(size_t)r * 6 + c - n3];
      }
      sB.push_back((float)v);
    }
  for (int r = 0; r < 6; ++r)
    for (int c = 0; c < ld; ++c) sG.push_back(c < n3 ? E[(size_t)c * 6 + r] : (c < n3 + 6 ? N[6 * r + c - n3] : 0.0));
  return nullptr;
}

// The grid as it is without bodies, after a failure while they were being
// replaced: no entry point may go on with sizes whose buffers are not there.
void forget_bodies(rbfib_grid* g) {
  g->nb = g->nbl = g->max_blobs = 0;
  g->h_boff.assign(1, 0);
  g->dense_body = g->dM_valid = g->dquat_valid = false;
  try {
    alloc_solver(g);
  } catch (CudaError&) {   // no memory for the fluid alone: need_solver reports it
  }
}

// Every entry point that solves or preconditions asks for its vectors first.
void need_solver(rbfib_grid* g) {
  const i64 n = g->n_total(), k = g->desc.precision == RBFIB_FP64 ? g->kr64.n : g->kr32.n;
  if (k < n || (i64)std::min({g->f32a.n, g->f32b.n, g->bvec.n, g->xvec.n, g->xrfd.n}) < n)
    throw CudaError{cudaErrorMemoryAllocation};
}

// ---------------------------------------------------------------- autotuner
// For each tunable kernel and grid shape, time every candidate block size
// (CUDA events on the grid's stream, best of a few launches) and keep the
// fastest.  Results are cached process-wide by shape, so a batch of many grids
// of a few sizes tunes each size once.
std::mutex g_tune_mu;
std::map<std::string, Tuning> g_tune_cache;

template <typename F>
int pick_block(cudaStream_t s, F launch) {
  const int cand[4] = {64, 128, 256, 512};
  cudaEvent_t e0, e1;
  ck(cudaEventCreate(&e0));
  ck(cudaEventCreate(&e1));
  int best = 256;
  float best_ms = 1e30f;
  for (int bs : cand) {
    launch(bs);   // warm-up
    float mn = 1e30f;
    for (int r = 0; r < 3; ++r) {
      ck(cudaEventRecord(e0, s));
      for (int k = 0; k < 4; ++k) launch(bs);
      ck(cudaEventRecord(e1, s));
      ck(cudaEventSynchronize(e1));
      float ms = 0.f;
      ck(cudaEventElapsedTime(&ms, e0, e1));
      mn = std::min(mn, ms);
    }
    if (mn < best_ms) { best_ms = mn; best = bs; }
  }
  cudaEventDestroy(e0);
  cudaEventDestroy(e1);
  return best;
}

void autotune(rbfib_grid* g) {
  const Dims& d = g->d;
  char key[160];
  std::snprintf(key, sizeof key, "%d,%d,%d,%d%d%d", d.n[0], d.n[1], d.n[2], d.per[0], d.per[1], d.per[2]);
  {
    std::lock_guard<std::mutex> lk(g_tune_mu);
    auto it = g_tune_cache.find(key);
    if (it != g_tune_cache.end()) { g->tune = it->second; return; }
  }
  Tuning t;
  if (g->nfl > (i64)8 * 1024 * 1024) {   // large grids are bandwidth-bound: keep 256
    g->tune = t;
    std::lock_guard<std::mutex> lk(g_tune_mu);
    g_tune_cache[key] = t;
    return;
  }
  double* x64 = g->xvec;
  double* y64 = g->bvec;
  float* x32 = g->f32a;
  float* y32 = g->f32b;
  ck(cudaMemsetAsync(x64, 0, sizeof(double) * g->nfl, g->s));
  ck(cudaMemsetAsync(x32, 0, sizeof(float) * g->nfl, g->s));
  ck(cudaMemsetAsync(y32, 0, sizeof(float) * g->nfl, g->s));
  const double eta = g->desc.eta;
  // the Stokes operator takes the block size only on non-uniform spacing (the
  // uniform-spacing kernels have fixed tile shapes): 0 = not tuned
  const bool uniform = d.h[0] == d.h[1] && d.h[1] == d.h[2];
  t.stokes64 = uniform ? 0 : pick_block(g->s, [&](int bs) {
    stokes_apply<double>(d, eta, x64, x64 + g->nf, y64, y64 + g->nf, g->s, bs);
  });
  t.stokes32 = uniform ? 0 : pick_block(g->s, [&](int bs) {
    stokes_apply<float>(d, (float)eta, x32, x32 + g->nf, y32, y32 + g->nf, g->s, bs);
  });
  // the smoothing sweeps only where the finest level has any (build_fd)
  if (g->fd_vel != 0)
    t.vrbgs = pick_block(g->s, [&](int bs) { vel_rbgs<float>(d, (float)eta, 0, x32, y32, g->s, bs); });
  if (g->fd_p != 0)
    t.prbgs = pick_block(g->s, [&](int bs) { p_rbgs<float>(d, 0, x32 + g->nf, y32 + g->nf, g->s, bs); });
  g->tune = t;
  std::lock_guard<std::mutex> lk(g_tune_mu);
  g_tune_cache[key] = t;
}

}  // namespace

// ======================================================================= ABI
extern "C" {

const char* rbfib_last_error(const rbfib_grid* g) { return g ? g->err.c_str() : "null grid"; }

uint64_t rbfib_launch_count(void) { return rbfib::g_launches.load(); }

int rbfib_body_block_info(const rbfib_grid* g, int32_t* dense, int64_t* warm_starts) {
  if (!g) return RBFIB_EINVAL;
  if (dense) *dense = g->dense_body ? 1 : 0;
  if (warm_starts) *warm_starts = g->ns_warm + g->ns_warm_dev;
  return RBFIB_OK;
}

int rbfib_step_mode(const rbfib_grid* g, int32_t* device_driven) {
  if (!g || !device_driven) return RBFIB_EINVAL;
  *device_driven = g->last_step_dev;
  return RBFIB_OK;
}

int rbfib_krylov_stats(const rbfib_grid* g, int64_t* iterations, int64_t* second_passes) {
  if (!g) return RBFIB_EINVAL;
  if (iterations) *iterations = g->gs_iters;
  if (second_passes) *second_passes = g->reorth_passes;
  return RBFIB_OK;
}

int rbfib_tuned_blocks(const rbfib_grid* g, int32_t out[4]) {
  if (!g || !out) return RBFIB_EINVAL;
  out[0] = g->tune.stokes64; out[1] = g->tune.stokes32; out[2] = g->tune.vrbgs; out[3] = g->tune.prbgs;
  return RBFIB_OK;
}

int rbfib_kernel_timer(rbfib_grid* g, int32_t which) {
  if (!g || which < 0 || which > 5) return RBFIB_EINVAL;
  try {
    ck(cudaStreamSynchronize(g->s));
  } catch (CudaError& e) {
    return fail(g, e.code, e.what());
  }
  g->timer_kind = which;
  g->tev_used = 0;
  g->timer_bytes = 0.0;
  g->timer_flops = 0.0;
  g->timer_launches = 0;
  return RBFIB_OK;
}

int rbfib_kernel_timer_overhead(rbfib_grid* g, int32_t reps, double* median_us) {
  if (!g || reps < 1 || reps > 10000 || !median_us) return RBFIB_EINVAL;
  std::vector<cudaEvent_t> ev;
  int st = RBFIB_OK;
  try {
    for (int i = 0; i < 2 * reps; ++i) {
      cudaEvent_t e;
      ck(cudaEventCreate(&e));
      ev.push_back(e);
    }
    // the same bracket as a timed launch: idle wait, event, launch, event
    for (int r = 0; r < reps; ++r) {
      gpu_delay(50000, g->s);
      ck(cudaEventRecord(ev[2 * r], g->s));
      gpu_empty(g->s);
      ck(cudaEventRecord(ev[2 * r + 1], g->s));
    }
    ck(cudaStreamSynchronize(g->s));
    std::vector<double> t(reps);
    for (int r = 0; r < reps; ++r) {
      float ms = 0.f;
      ck(cudaEventElapsedTime(&ms, ev[2 * r], ev[2 * r + 1]));
      t[r] = 1000.0 * ms;
    }
    std::sort(t.begin(), t.end());
    *median_us = t[reps / 2];
  } catch (CudaError& e) {
    st = fail(g, e.code, e.what());
  }
  for (cudaEvent_t e : ev) cudaEventDestroy(e);
  return st;
}

int rbfib_kernel_timer_read(rbfib_grid* g, double* total_ms, int64_t* launches, double* alg_bytes, double* alg_flops) {
  if (!g) return RBFIB_EINVAL;
  double tot = 0.0;
  try {
    ck(cudaStreamSynchronize(g->s));
    for (size_t i = 0; i + 1 < g->tev_used; i += 2) {
      float ms = 0.f;
      ck(cudaEventElapsedTime(&ms, g->tev[i], g->tev[i + 1]));
      tot += ms;
    }
  } catch (CudaError& e) {
    return fail(g, e.code, e.what());
  }
  if (total_ms) *total_ms = tot;
  if (launches) *launches = g->timer_launches;
  if (alg_bytes) *alg_bytes = g->timer_bytes;
  if (alg_flops) *alg_flops = g->timer_flops;
  return RBFIB_OK;
}

}  // extern "C"

// Used by the ensemble work queue between calls: every call on a grid ends
// with its stream synchronised, so the next call may run on another stream.
void rbfib_grid_bind_stream(rbfib_grid* g, cudaStream_t s) { g->s = s; }



extern "C" {

int rbfib_create_grid(const rbfib_grid_desc* desc, void* stream, rbfib_grid** out) {
  if (!desc || !out) return RBFIB_EINVAL;
  *out = nullptr;
  const rbfib_grid_desc& D = *desc;
  for (int a = 0; a < 3; ++a)
    if (D.n[a] < 2 || (D.periodic[a] != 0 && D.periodic[a] != 1)) return RBFIB_EINVAL;
  if (D.periodic[0] && D.periodic[1] && D.periodic[2]) return RBFIB_EINVAL;
  if (!(D.h > 0) || !(D.eta > 0) || (D.kernel != 3 && D.kernel != 6) || D.restart < 1 || D.restart > 64 || D.max_iter < 1 ||
      !(D.rtol > 0) || (D.precision != RBFIB_FP64 && D.precision != RBFIB_FP32_REFINED))
    return RBFIB_EINVAL;
  for (int a = 0; a < 3; ++a)
    if (D.wall_vel[2 * a][a] != 0.0 || D.wall_vel[2 * a + 1][a] != 0.0) return RBFIB_EINVAL;
  // free-slip walls: flags 0 / 1, no wall velocity, and no velocity component
  // left without a no-slip wall (a constant null mode of its viscous operator)
  for (int w = 0; w < 6; ++w) {
    if (D.free_slip[w] != 0 && D.free_slip[w] != 1) return RBFIB_EINVAL;
    if (D.free_slip[w] && !D.periodic[w / 2])
      for (int c = 0; c < 3; ++c)
        if (D.wall_vel[w][c] != 0.0) return RBFIB_EINVAL;
  }
  for (int a = 0; a < 3; ++a) {
    if (!D.periodic[a]) continue;
    bool pinned = false;
    for (int b = 0; b < 3; ++b)
      if (b != a && !D.periodic[b] && !(D.free_slip[2 * b] && D.free_slip[2 * b + 1])) pinned = true;
    if (!pinned) return RBFIB_EINVAL;
  }
  rbfib_grid* g = new rbfib_grid();
  try {
    g->desc = D;
    g->s = (cudaStream_t)stream;
    build_levels(g);
    build_fd(g);
    g->levels[0].d.kw = D.kernel;
    g->d = g->levels[0].d;
    for (int w = 0; w < 6; ++w)
      for (int c = 0; c < 3; ++c) {
        g->walls.v[w][c] = D.wall_vel[w][c];
        if (D.wall_vel[w][c] != 0.0) g->walls_move = true;
      }
    g->nf = g->d.fo[3];
    g->nc = g->d.nc;
    g->nfl = g->nf + g->nc;
    g->dV = D.h * D.h * D.h;
    g->kappa = pressure_kappa(g->d);
    g->pair = pair_mobility(D.kernel);
    build_stress_layout(g);
    g->nparts = 152 * 4;
    g->part.alloc(part_buffer_doubles(g->nparts));
    ck(cudaMemsetAsync(g->part.p, 0, sizeof(double) * part_buffer_doubles(g->nparts), g->s));
    g->small.alloc((size_t)(D.restart + 1) * D.restart + 4 * D.restart + 512);
    ck(cudaMallocHost((void**)&g->h_pinned, 64 * sizeof(double)));
    g->gst.alloc(8);
    g->dpar.alloc(8);
    g->dstep.alloc(4);
    g->dinfo.alloc(32);
    g->drsi.alloc(8);
    g->drel.alloc(8);
    g->drst.alloc(8);
    g->dwarm.alloc(1);
    ck(cudaMemsetAsync(g->dwarm.p, 0, sizeof(long long), g->s));
    if (const char* e = std::getenv("RBFIB_NO_GRAPHS")) g->use_graphs = (e[0] == '0');
    if (const char* e = std::getenv("RBFIB_NO_STEP_GRAPH")) g->step_graphs = (e[0] == '0');
    g->mg32.build(g->levels);
    g->bcount.alloc(g->nc + 1);
    g->bfill.alloc(g->nc);
    g->celloff.alloc(g->nc + 1);
    g->bbsum.alloc((g->nc + 1) / 1024 + 2);
    g->boff.alloc(1);
    ck(cudaMemsetAsync(g->boff, 0, sizeof(int), g->s));
    g->h_boff.assign(1, 0);
    g->fnoise.alloc(g->nf);
    g->Wst.alloc(g->stress.total);
    alloc_solver(g);
    autotune(g);
    ck(cudaStreamSynchronize(g->s));
  } catch (CudaError& e) {
    std::string msg = std::string("create_grid: ") + e.what();
    delete g;
    (void)msg;
    return RBFIB_ECUDA;
  }
  *out = g;
  return RBFIB_OK;
}

void rbfib_destroy(rbfib_grid* g) {
  if (!g) return;
  if (g->s) cudaStreamSynchronize(g->s);
  for (cudaEvent_t e : g->tev) cudaEventDestroy(e);
  drop_graphs(g);
  if (g->h_pinned) cudaFreeHost(g->h_pinned);
  for (cudaStream_t& cs : g->cap_streams)
    if (cs) cudaStreamDestroy(cs);
  delete g;
}

int rbfib_saddle_layout(const rbfib_grid* g, int64_t off[7]) {
  if (!g || !off) return RBFIB_EINVAL;
  off[0] = 0;
  off[1] = g->d.fo[1];
  off[2] = g->d.fo[2];
  off[3] = g->nf;
  off[4] = g->nfl;
  off[5] = g->nfl + 3 * (i64)g->nbl;
  off[6] = off[5] + 6 * (i64)g->nb;
  return RBFIB_OK;
}

int rbfib_set_bodies(rbfib_grid* g, int32_t n_bodies, const int32_t* blob_offsets, const double* ref_blobs,
                     const double* q, const double* quat) {
  if (!g || n_bodies < 0 || (n_bodies > 0 && (!blob_offsets || !ref_blobs || !q || !quat)))
    return fail(g, RBFIB_EINVAL, "set_bodies: bad arguments");
  bool replaced = false;   // whether the grid's previous bodies are gone
  try {
    std::vector<int> off(n_bodies + 1, 0);
    if (n_bodies > 0) {
      std::memcpy(off.data(), blob_offsets, sizeof(int) * (n_bodies + 1));
      if (off[0] != 0) return fail(g, RBFIB_EINVAL, "set_bodies: blob_offsets[0] must be 0");
      for (int p = 0; p < n_bodies; ++p)
        if (off[p + 1] <= off[p]) return fail(g, RBFIB_EINVAL, "set_bodies: every body needs at least one blob");
    }
    // all that can be refused is looked at before any state of the grid changes
    const int nb = n_bodies, nbl = off[n_bodies];
    std::vector<double> ref(3 * (size_t)nbl);
    if (nb > 0) {
      if (cudaStreamSynchronize(g->s) != cudaSuccess ||
          cudaMemcpy(ref.data(), ref_blobs, sizeof(double) * ref.size(), cudaMemcpyDeviceToHost) != cudaSuccess)
        return fail(g, RBFIB_ECUDA, "set_bodies: cannot read ref_blobs");
      // a rigid body needs three blobs off one line: with collinear blobs the
      // rotation about their line is undetermined and the system is singular
      for (int p = 0; p < nb; ++p) {
        const double* r0 = &ref[3 * (size_t)off[p]];
        double u[3] = {0, 0, 0}, un = 0.0;
        for (int i = off[p] + 1; i < off[p + 1]; ++i) {
          const double* r = &ref[3 * (size_t)i];
          const double d2 = (r[0] - r0[0]) * (r[0] - r0[0]) + (r[1] - r0[1]) * (r[1] - r0[1]) +
                            (r[2] - r0[2]) * (r[2] - r0[2]);
          if (d2 > un) { un = d2; for (int a = 0; a < 3; ++a) u[a] = r[a] - r0[a]; }
        }
        double worst = 0.0;
        for (int i = off[p] + 1; i < off[p + 1] && un > 0.0; ++i) {
          const double* r = &ref[3 * (size_t)i];
          const double dv[3] = {r[0] - r0[0], r[1] - r0[1], r[2] - r0[2]};
          const double cx = dv[1] * u[2] - dv[2] * u[1], cy = dv[2] * u[0] - dv[0] * u[2], cz = dv[0] * u[1] - dv[1] * u[0];
          worst = std::max(worst, std::sqrt(cx * cx + cy * cy + cz * cz) / un);
        }
        if (!(worst > 1e-9)) return fail(g, RBFIB_EINVAL, "set_bodies: a body's blobs lie on one line");
      }
    }
    // body lengths and shape table
    std::vector<double> Lp(std::max(nb, 1), 0.0);
    std::vector<int> shape_of(std::max(nb, 1), 0), shape_rep;
    int max_blobs = 0;
    for (int p = 0; p < nb; ++p) {
      const int n = off[p + 1] - off[p];
      max_blobs = std::max(max_blobs, n);
      const double* x = ref.data() + 3 * (size_t)off[p];
      double mx = 0.0;
      for (int i = 0; i < n; ++i)
        for (int j = i + 1; j < n; ++j) {
          double dd = 0.0;
          for (int a = 0; a < 3; ++a) dd += (x[3 * i + a] - x[3 * j + a]) * (x[3 * i + a] - x[3 * j + a]);
          mx = std::max(mx, std::sqrt(dd));
        }
      Lp[p] = mx;
      int found = -1;
      for (size_t s = 0; s < shape_rep.size(); ++s) {
        const int q0 = shape_rep[s];
        if (off[q0 + 1] - off[q0] == n &&
            std::memcmp(ref.data() + 3 * (size_t)off[q0], x, sizeof(double) * 3 * n) == 0) { found = (int)s; break; }
      }
      if (found < 0) { found = (int)shape_rep.size(); shape_rep.push_back(p); }
      shape_of[p] = found;
    }
    // coupled body block when every blob pair fits a small dense matrix, else
    // per-shape body-block matrices in the body frame (k_body.cu)
    const bool dense = nb >= 2 && 3 * nbl <= kDenseBodyMaxRows && 6 * nb <= kDenseBodyMaxBodyRows;
    const int ns = (int)shape_rep.size();
    std::vector<i64> soff(std::max(ns, 1), 0), soffg(std::max(ns, 1), 0);
    std::vector<float> sB;
    std::vector<double> sG;
    for (int s = 0; s < ns && !dense; ++s) {
      const int p = shape_rep[s];
      soff[s] = (i64)sB.size();
      soffg[s] = (i64)sG.size();
      if (const char* why = shape_matrix(g, ref.data() + 3 * (size_t)off[p], off[p + 1] - off[p], sB, sG))
        return fail(g, RBFIB_EINVAL, std::string("set_bodies: ") + why);
    }

    ck(cudaStreamSynchronize(g->s));
    drop_graphs(g);
    replaced = true;
    g->nb = nb;
    g->nbl = nbl;
    g->h_boff = off;
    g->max_blobs = max_blobs;
    g->dense_body = dense;
    g->dM_valid = false;
    g->dquat_valid = false;
    g->boff.alloc(nb + 1);
    ck(cudaMemcpyAsync(g->boff, off.data(), sizeof(int) * (nb + 1), cudaMemcpyHostToDevice, g->s));
    std::vector<int> bob(nbl);
    for (int p = 0; p < nb; ++p)
      for (int i = off[p]; i < off[p + 1]; ++i) bob[i] = p;
    g->bob.alloc(std::max(nbl, 1));
    if (nbl) ck(cudaMemcpyAsync(g->bob, bob.data(), sizeof(int) * nbl, cudaMemcpyHostToDevice, g->s));
    g->ref.alloc(3 * (size_t)std::max(nbl, 1));
    if (nbl) ck(cudaMemcpyAsync(g->ref, ref_blobs, sizeof(double) * 3 * nbl, cudaMemcpyDeviceToDevice, g->s));
    for (Config* c : {&g->cur, &g->plus, &g->minus, &g->next}) alloc_config(g, *c);
    if (nb) {
      ck(cudaMemcpyAsync(g->cur.q, q, sizeof(double) * 3 * nb, cudaMemcpyDeviceToDevice, g->s));
      ck(cudaMemcpyAsync(g->cur.quat, quat, sizeof(double) * 4 * nb, cudaMemcpyDeviceToDevice, g->s));
    }
    g->bkey.alloc(std::max(nbl, 1));
    if (dense) {
      g->dM.alloc((size_t)9 * nbl * nbl);
      g->dMw.alloc((size_t)9 * nbl * nbl);
      g->dTw.alloc((size_t)9 * nbl * nbl);
      g->dUw.alloc((size_t)9 * nbl * nbl);
      g->dss.alloc(1);
      g->dquat.alloc(4 * (size_t)nb);
      g->dP.alloc((size_t)18 * nbl * nb);
      g->dE.alloc((size_t)18 * nbl * nb);
      g->dB.alloc((size_t)3 * nbl * body_ld(3 * nbl + 6 * nb));
      g->dG.alloc((size_t)6 * nb * body_ld(3 * nbl + 6 * nb));
      g->dN.alloc((size_t)36 * nb * nb);
      g->dNw.alloc((size_t)72 * nb * nb);
      g->dstatus.alloc(1);
    }
    g->Lp.alloc(std::max(nb, 1));
    ck(cudaMemcpyAsync(g->Lp, Lp.data(), sizeof(double) * std::max(nb, 1), cudaMemcpyHostToDevice, g->s));
    g->shape_of.alloc(std::max(nb, 1));
    ck(cudaMemcpyAsync(g->shape_of, shape_of.data(), sizeof(int) * std::max(nb, 1), cudaMemcpyHostToDevice, g->s));
    g->shape_off.alloc(std::max(ns, 1));
    ck(cudaMemcpyAsync(g->shape_off, soff.data(), sizeof(i64) * std::max(ns, 1), cudaMemcpyHostToDevice, g->s));
    g->shape_B.alloc(std::max<size_t>(sB.size(), 1));
    if (!sB.empty())
      ck(cudaMemcpyAsync(g->shape_B, sB.data(), sizeof(float) * sB.size(), cudaMemcpyHostToDevice, g->s));
    g->shape_offg.alloc(std::max(ns, 1));
    ck(cudaMemcpyAsync(g->shape_offg, soffg.data(), sizeof(i64) * std::max(ns, 1), cudaMemcpyHostToDevice, g->s));
    g->shape_G.alloc(std::max<size_t>(sG.size(), 1));
    if (!sG.empty())
      ck(cudaMemcpyAsync(g->shape_G, sG.data(), sizeof(double) * sG.size(), cudaMemcpyHostToDevice, g->s));
    ck(cudaStreamSynchronize(g->s));
    // body-sized work arrays
    const size_t b6 = 6 * (size_t)std::max(nb, 1), l3 = 3 * (size_t)std::max(nbl, 1);
    for (DBuf<double>* b : {&g->bodyF, &g->bodyW, &g->bodyWn}) b->alloc(b6);
    g->blobS.alloc(l3);
    alloc_solver(g);
    refresh_config(g, g->cur, true);
    ck(cudaStreamSynchronize(g->s));
    ck(cudaGetLastError());
  } catch (CudaError& e) {
    if (replaced) forget_bodies(g);
    return fail(g, e.code, std::string("set_bodies: ") + e.what());
  } catch (std::exception& e) {
    if (replaced) forget_bodies(g);
    return fail(g, RBFIB_EINTERNAL, std::string("set_bodies: ") + e.what());
  }
  return RBFIB_OK;
}

int rbfib_apply_preconditioner(rbfib_grid* g, const double* r, double* z) {
  if (!g || !r || !z) return fail(g, RBFIB_EINVAL, "apply_preconditioner: null argument");
  try {
    need_solver(g);
    convert<double, float>(r, g->f32a, g->n_total(), g->s);
    precond<float>(g, g->f32a, g->f32b, true, z, 0.0);
    ck(cudaGetLastError());
  } catch (CudaError& e) {
    return fail(g, e.code, std::string("apply_preconditioner: ") + e.what());
  }
  return RBFIB_OK;
}

int rbfib_apply_saddle(rbfib_grid* g, const void* x, void* y, int32_t dtype) {
  if (!g || !x || !y) return fail(g, RBFIB_EINVAL, "apply_saddle: null argument");
  try {
    if (dtype == RBFIB_DTYPE_F64) apply_A<double>(g, (const double*)x, (double*)y, true);
    else if (dtype == RBFIB_DTYPE_F32) apply_A<float>(g, (const float*)x, (float*)y, true);
    else return fail(g, RBFIB_EINVAL, "apply_saddle: dtype");
    ck(cudaGetLastError());
  } catch (CudaError& e) {
    return fail(g, e.code, std::string("apply_saddle: ") + e.what());
  }
  return RBFIB_OK;
}

}  // extern "C"

namespace {

// Graph-captured restart cycles unless disabled or a kernel timer is active
// (event records cannot sit inside conditional graph bodies).
bool use_graph_path(rbfib_grid* g) { return g->use_graphs && g->timer_kind == 0; }

// Right-hand side of the constrained system: fluid forcing + wall terms,
// -slip + J wall part, forces.  b is FP64 in the saddle layout.
void build_rhs(rbfib_grid* g, const double* FT, const double* slip, const double* fluid, bool walls, double* b) {
  const i64 n = g->n_total();
  need_solver(g);
  ck(cudaMemsetAsync(b, 0, sizeof(double) * n, g->s));
  if (fluid) ck(cudaMemcpyAsync(b, fluid, sizeof(double) * g->nf, cudaMemcpyDeviceToDevice, g->s));
  if (walls && g->walls_move) wall_rhs<double>(g->d, g->walls, g->desc.eta, b, g->s);
  if (g->nbl > 0) {
    double* bl = b + g->nfl;
    if (walls && g->walls_move) interp_walls(g->d, g->walls, g->nbl, g->cur.r, 0.0, bl, g->s);
    if (slip) axpby<double>(bl, slip, -1.0, 1.0, 3 * (i64)g->nbl, g->s);
  }
  if (g->nb > 0 && FT)
    ck(cudaMemcpyAsync(b + g->nfl + 3 * (i64)g->nbl, FT, sizeof(double) * 6 * g->nb, cudaMemcpyDeviceToDevice, g->s));
}

// ------------------------------------------------- device-driven solves
// Captured on g->s (the step graph being built): no host reads.  The restart
// cycles of a solve run in a WHILE node whose condition the check after each
// cycle sets; info / rel receive iterations, status, cycles, second passes
// and the true relative residual.  rtol_p / maxit_p (device, may be null)
// override rtol / maxit (the refinement's inner solves).
// Returns the launches captured in the WHILE body; per_iter (may be null)
// receives one iteration's launches with its gated second pass.
template <typename T>
long long solve_dev(rbfib_grid* g, const T* b, T* x, bool wb, double rtol, int maxit, const double* rtol_p,
                    const int* maxit_p, int* info, double* rel, long long* per_iter) {
  KrylovStore<T>& K = kr_of<T>(g);
  const i64 n = wb ? g->n_total() : g->nfl, ld = K.n, nfl = g->nfl;
  multi_dot<T>(b, b, ld, 1, n, nfl, g->dV, g->part, g->nparts, g->dpar + 3, g->s);
  ck(cudaMemsetAsync(x, 0, sizeof(T) * n, g->s));
  ck(cudaMemcpyAsync(K.w, b, sizeof(T) * n, cudaMemcpyDeviceToDevice, g->s));
  const cudaGraphConditionalHandle h = new_handle(g, 0u);
  solve_init(g->dpar, g->gst, rtol, maxit, rtol_p, maxit_p, h, info, rel, g->s);
  const long long a0 = rbfib::g_launches.load();
  cond_node(g, h, cudaGraphCondTypeWhile, 1, [&](int) {
    capture_cycle<T>(g, b, x, wb, per_iter);
    solve_check(g->dpar, g->gst, h, info, rel, g->s);
  });
  return (long long)rbfib::g_launches.load() - a0;
}

// FP32 kernels inside FP64 refinement, device-driven: the sweeps run in a
// WHILE node around the inner FP32 solve's own WHILE node.
long long refine_dev(rbfib_grid* g, const double* b, double* x, bool wb, int* info, double* rel, long long* per_iter) {
  const i64 n = wb ? g->n_total() : g->nfl;
  const double rtol = g->desc.rtol;
  double* r = g->rres;
  int* inner = g->dinfo.p + 16;
  multi_dot<double>(b, b, n, 1, n, g->nfl, g->dV, g->part, g->nparts, g->drst.p + 0, g->s);
  ck(cudaMemsetAsync(x, 0, sizeof(double) * n, g->s));
  ck(cudaMemcpyAsync(r, b, sizeof(double) * n, cudaMemcpyDeviceToDevice, g->s));
  const cudaGraphConditionalHandle h = new_handle(g, 0u);
  refine_init(g->drst, g->drsi, h, info, rel, g->s);
  const long long a0 = rbfib::g_launches.load();
  cond_node(g, h, cudaGraphCondTypeWhile, 1, [&](int) {
    refine_sweep(g->drst, g->drsi, rtol, kInnerTol, g->desc.max_iter, kr_of<float>(g).m, g->s);
    convert<double, float>(r, g->f32a, n, g->s);
    solve_dev<float>(g, g->f32a, g->f32b, wb, 0.0, 0, g->drst.p + 2, g->drsi.p + 3, inner, g->drel.p + 3,
                     per_iter);
    convert<float, double>(g->f32b, r, n, g->s);
    axpby<double>(x, r, 1.0, 1.0, n, g->s);
    apply_A<double>(g, x, r, wb);
    axpby<double>(r, b, 1.0, -1.0, n, g->s);
    multi_dot<double>(r, r, n, 1, n, g->nfl, g->dV, g->part, g->nparts, g->drst.p + 3, g->s);
    refine_check(g->drst.p + 3, g->drst, g->drsi, inner, rtol, g->desc.max_iter, h, info, rel, g->s);
  });
  return (long long)rbfib::g_launches.load() - a0;
}

// Solve A x = b (FP64 in and out).  FP64 mode: FGMRES in FP64.  FP32 mode:
// iterative refinement, r = b - A x in FP64, inner FGMRES in FP32.  While the
// device-driven step is captured (g->dev), the solve is captured instead,
// reporting into slot `which` of dinfo / drel.
int solve_system(rbfib_grid* g, const double* b, double* x, bool with_bodies, rbfib_solve_info* info,
                 int which = -1) {
  if (g->dev) {
    int* di = g->dinfo.p + 4 * which;
    double* dr = g->drel.p + which;
    long long per_iter = 0, body = 0;
    if (g->desc.precision == RBFIB_FP64)
      body = solve_dev<double>(g, b, x, with_bodies, g->desc.rtol, g->desc.max_iter, nullptr, nullptr, di, dr,
                               &per_iter);
    else
      body = refine_dev(g, b, x, with_bodies, di, dr, &per_iter);
    // one pass of the WHILE body: its fixed part plus one captured iteration
    g->cap_body_fixed[which] = body - per_iter;
    g->cap_per_iter[which] = per_iter;
    g->cap_bodies += body;
    project_mean(x + g->nf, g->nc, g->part, g->nparts, g->s);
    return 0;
  }
  const i64 n = with_bodies ? g->n_total() : g->nfl;
  const double rtol = g->desc.rtol;
  int iters = 0, st = 0;
  double rel = 0.0;
  if (g->desc.precision == RBFIB_FP64) {
    st = use_graph_path(g) ? fgmres_graph<double>(g, b, x, with_bodies, rtol, g->desc.max_iter, iters, rel)
                           : fgmres<double>(g, b, x, with_bodies, rtol, g->desc.max_iter, iters, rel);
    if (info) { info->iterations = iters; info->refinements = 0; info->rel_residual = rel; }
  } else {
    // outer refinement in FP64
    SmallPtrs sp = small_ptrs(g, g->desc.restart);
    double* r = g->rres;      // FP64 residual of the refinement
    multi_dot<double>(b, b, n, 1, n, g->nfl, g->dV, g->part, g->nparts, sp.bn, g->s);
    const double bn = std::sqrt(std::max(read_scalar(g, sp.bn), 0.0));
    ck(cudaMemsetAsync(x, 0, sizeof(double) * n, g->s));
    if (!(bn > 0.0)) { if (info) { info->iterations = 0; info->refinements = 0; info->rel_residual = 0; } return 0; }
    ck(cudaMemcpyAsync(r, b, sizeof(double) * n, cudaMemcpyDeviceToDevice, g->s));
    int sweeps = 0, total = 0;
    rel = 1.0;
    // Each FP32 sweep asks for a reduction of inner_tol relative to its own
    // right-hand side, but at most the remaining factor to rtol (halved,
    // so the last sweep lands below it), and runs at most one restart
    // cycle: an FP32 solve whose residual estimate stalls near FP32
    // roundoff then hands back after m iterations instead of running on.
    // Measured on the two-sphere SEM step (iterations of the three solves,
    // steps/s): 1e-4: 39/19/38, 76.5; 1e-5: 43/21/41, 71.9; 1e-6: 39/20/40,
    // 73.6 (every solve takes two sweeps in each case).
    const double inner_tol = kInnerTol;
    const int inner_cap = kr_of<float>(g).m;
    while (rel > rtol && total < g->desc.max_iter && sweeps < 50) {
      convert<double, float>(r, g->f32a, n, g->s);
      int it = 0;
      double irel = 0.0;
      const double tol_s = std::max(inner_tol, 0.5 * rtol / rel);
      const int cap = std::min(g->desc.max_iter - total, inner_cap);
      int ist = use_graph_path(g)
                    ? fgmres_graph<float>(g, g->f32a, g->f32b, with_bodies, tol_s, cap, it, irel)
                    : fgmres<float>(g, g->f32a, g->f32b, with_bodies, tol_s, cap, it, irel);
      total += it;
      ++sweeps;
      if (ist == RBFIB_ENAN) { st = ist; break; }
      // x += d (FP64), r = b - A x (FP64)
      convert<float, double>(g->f32b, r, n, g->s);
      axpby<double>(x, r, 1.0, 1.0, n, g->s);
      apply_A<double>(g, x, r, with_bodies);
      axpby<double>(r, b, 1.0, -1.0, n, g->s);
      multi_dot<double>(r, r, n, 1, n, g->nfl, g->dV, g->part, g->nparts, sp.bn, g->s);
      rel = std::sqrt(std::max(read_scalar(g, sp.bn), 0.0)) / bn;
      if (std::isnan(rel)) { st = RBFIB_ENAN; break; }
    }
    if (st == 0 && rel > rtol) st = RBFIB_ENOCONV;
    if (info) { info->iterations = total; info->refinements = sweeps; info->rel_residual = rel; }
  }
  // pressure gauge: mean(pi) = 0
  project_mean(x + g->nf, g->nc, g->part, g->nparts, g->s);
  return st;
}

}  // namespace

extern "C" {

int rbfib_mobility_solve(rbfib_grid* g, const double* FT, const double* slip, const double* fluid_rhs, double* U,
                         double* x_full, rbfib_solve_info* info) {
  if (!g || (g->nb > 0 && !FT)) return fail(g, RBFIB_EINVAL, "mobility_solve: null argument");
  try {
    build_rhs(g, FT, slip, fluid_rhs, true, g->bvec);
    int st = solve_system(g, g->bvec, g->xvec, true, info);
    if (U && g->nb > 0)
      ck(cudaMemcpyAsync(U, g->xvec.p + g->nfl + 3 * (i64)g->nbl, sizeof(double) * 6 * g->nb,
                         cudaMemcpyDeviceToDevice, g->s));
    if (x_full) ck(cudaMemcpyAsync(x_full, g->xvec, sizeof(double) * g->n_total(), cudaMemcpyDeviceToDevice, g->s));
    ck(cudaStreamSynchronize(g->s));
    ck(cudaGetLastError());
    if (st) return fail(g, st, st == RBFIB_ENOCONV ? "mobility_solve: no convergence" : "mobility_solve: NaN");
  } catch (CudaError& e) {
    return fail(g, e.code, std::string("mobility_solve: ") + e.what());
  }
  return RBFIB_OK;
}

int rbfib_stokes_solve(rbfib_grid* g, const double* f, double* v, double* pi, rbfib_solve_info* info) {
  if (!g || !f || !v) return fail(g, RBFIB_EINVAL, "stokes_solve: null argument");
  try {
    need_solver(g);
    ck(cudaMemsetAsync(g->bvec, 0, sizeof(double) * g->nfl, g->s));
    ck(cudaMemcpyAsync(g->bvec, f, sizeof(double) * g->nf, cudaMemcpyDeviceToDevice, g->s));
    int st = solve_system(g, g->bvec, g->xvec, false, info);
    ck(cudaMemcpyAsync(v, g->xvec, sizeof(double) * g->nf, cudaMemcpyDeviceToDevice, g->s));
    if (pi) ck(cudaMemcpyAsync(pi, g->xvec.p + g->nf, sizeof(double) * g->nc, cudaMemcpyDeviceToDevice, g->s));
    ck(cudaStreamSynchronize(g->s));
    ck(cudaGetLastError());
    if (st) return fail(g, st, "stokes_solve: no convergence");
  } catch (CudaError& e) {
    return fail(g, e.code, std::string("stokes_solve: ") + e.what());
  }
  return RBFIB_OK;
}

int rbfib_binning(rbfib_grid* g, int32_t* perm, int32_t* cell_offsets) {
  if (!g) return RBFIB_EINVAL;
  try {
    if (perm && g->nbl) ck(cudaMemcpyAsync(perm, g->cur.perm, sizeof(int) * g->nbl, cudaMemcpyDeviceToDevice, g->s));
    if (cell_offsets)
      ck(cudaMemcpyAsync(cell_offsets, g->celloff, sizeof(int) * (g->nc + 1), cudaMemcpyDeviceToDevice, g->s));
    ck(cudaGetLastError());
  } catch (CudaError& e) {
    return fail(g, e.code, std::string("binning: ") + e.what());
  }
  return RBFIB_OK;
}

int rbfib_blob_positions(rbfib_grid* g, double* r) {
  if (!g || !r) return RBFIB_EINVAL;
  try {
    if (g->nbl) ck(cudaMemcpyAsync(r, g->cur.r, sizeof(double) * 3 * g->nbl, cudaMemcpyDeviceToDevice, g->s));
  } catch (CudaError& e) {
    return fail(g, e.code, e.what());
  }
  return RBFIB_OK;
}

int rbfib_philox_words(rbfib_grid* g, uint64_t seed, uint64_t step, uint32_t attempt, uint32_t purpose,
                       uint64_t first_block, int64_t n_blocks, uint64_t* out) {
  if (!g || n_blocks < 0 || (n_blocks > 0 && (!out || (reinterpret_cast<uintptr_t>(out) & 15))))
    return fail(g, RBFIB_EINVAL, "philox_words: bad argument");
  try {
    philox_words(seed, step, attempt, purpose, first_block, n_blocks, (unsigned long long*)out, g->s);
    ck(cudaGetLastError());
  } catch (CudaError& e) {
    return fail(g, e.code, e.what());
  }
  return RBFIB_OK;
}

int rbfib_philox_normals(rbfib_grid* g, uint64_t seed, uint64_t step, uint32_t attempt, uint32_t purpose,
                         int64_t count, double* out) {
  if (!g || count < 0 || (count > 0 && !out)) return fail(g, RBFIB_EINVAL, "philox_normals: bad argument");
  try {
    philox_normals(seed, step, attempt, purpose, count, out, g->s);
    ck(cudaGetLastError());
  } catch (CudaError& e) {
    return fail(g, e.code, e.what());
  }
  return RBFIB_OK;
}

int rbfib_stochastic_forcing(rbfib_grid* g, double kT, double dt, uint64_t seed, uint64_t step, uint32_t attempt,
                             double* out) {
  if (!g || !out || !(dt > 0) || !(kT >= 0)) return fail(g, RBFIB_EINVAL, "stochastic_forcing: bad argument");
  try {
    philox_normals(seed, step, attempt, 1u, g->stress.total, g->Wst, g->s);
    const double c = std::sqrt(2.0 * g->desc.eta * kT / (g->dV * dt));
    stress_divergence(g->d, g->stress, g->Wst, c, out, g->s);
    ck(cudaGetLastError());
  } catch (CudaError& e) {
    return fail(g, e.code, e.what());
  }
  return RBFIB_OK;
}

int rbfib_spread(rbfib_grid* g, const double* lambda, double* f) {
  if (!g || !f || (g->nbl && !lambda)) return fail(g, RBFIB_EINVAL, "spread: null argument");
  try {
    ck(cudaMemsetAsync(f, 0, sizeof(double) * g->nf, g->s));
    spread_tab(g->d, view_of(g, g->cur), lambda, 1.0 / g->dV, f, g->s);
    ck(cudaGetLastError());
  } catch (CudaError& e) {
    return fail(g, e.code, e.what());
  }
  return RBFIB_OK;
}

int rbfib_interpolate(rbfib_grid* g, const double* v, double* u, int32_t with_walls) {
  if (!g || !v || (g->nbl && !u)) return fail(g, RBFIB_EINVAL, "interpolate: null argument");
  try {
    interp_tab(g->d, view_of(g, g->cur), v, 1.0, 0.0, u, g->s);
    if (with_walls && g->walls_move) interp_walls(g->d, g->walls, g->nbl, g->cur.r, 1.0, u, g->s);
    ck(cudaGetLastError());
  } catch (CudaError& e) {
    return fail(g, e.code, e.what());
  }
  return RBFIB_OK;
}

}  // extern "C"

namespace {
Potentials potentials_of(const rbfib_sem_params* p) {
  Potentials P;
  P.gravity = p->gravity;
  P.blob_g = p->blob_gravity;
  P.pair_phi0 = p->pair_phi0; P.pair_b = p->pair_b; P.pair_d = p->pair_d;
  P.wall_phi0 = p->wall_phi0; P.wall_b = p->wall_b; P.wall_d = p->wall_d;
  P.bw_phi0 = p->blob_wall_phi0; P.bw_b = p->blob_wall_b; P.bw_d = p->blob_wall_d;
  P.yuk_u0 = p->yukawa_u0; P.yuk_dh = p->yukawa_dh; P.yuk_lambda = p->yukawa_lambda;
  P.sub_u0 = p->substrate_u0; P.sub_s = p->substrate_s;
  return P;
}

}  // namespace

extern "C" {

int rbfib_body_forces(rbfib_grid* g, const rbfib_sem_params* p, double* out) {
  if (!g || !p || (g->nb && !out)) return fail(g, RBFIB_EINVAL, "body_forces: null argument");
  try {
    body_forces(g->d, potentials_of(p), view_of(g, g->cur), p->force_ext, out, g->s);
    ck(cudaGetLastError());
  } catch (CudaError& e) {
    return fail(g, e.code, e.what());
  }
  return RBFIB_OK;
}

int rbfib_set_blob_positions(rbfib_grid* g, const double* r) {
  if (!g || (g->nbl > 0 && !r)) return fail(g, RBFIB_EINVAL, "set_blob_positions: null argument");
  try {
    if (g->nbl) ck(cudaMemcpyAsync(g->cur.r, r, sizeof(double) * 3 * g->nbl, cudaMemcpyDeviceToDevice, g->s));
    arms_from_positions(g->nbl, g->bob, g->cur.r, g->cur.q, g->cur.arm, g->s);
    binning(g->d, g->nbl, g->cur.r, g->cur.perm, g->celloff, g->bkey, g->bcount, g->bfill, g->bbsum, g->s);
    stencil_build(g->d, g->nbl, g->cur.r, g->cur.st64, g->cur.st32, g->s);
    if (g->dense_body) build_body_block(g, g->cur.r, g->cur.arm, nullptr);
    ck(cudaGetLastError());
  } catch (CudaError& e) {
    return fail(g, e.code, e.what());
  }
  return RBFIB_OK;
}

int rbfib_mobility_solve_adjoint(rbfib_grid* g, const double* dL_dU, const double* x_fwd, double* dL_dr,
                                 double* dL_dslip, rbfib_solve_info* info) {
  if (!g || !dL_dU || !x_fwd) return fail(g, RBFIB_EINVAL, "mobility_solve_adjoint: null argument");
  for (int w = 0; w < 6; ++w)
    for (int c = 0; c < 3; ++c)
      if (g->walls.v[w][c] != 0.0) return fail(g, RBFIB_EINVAL, "mobility_solve_adjoint: moving walls");
  try {
    const i64 n = g->n_total();
    // A z = [0, 0, 0, dL/dU]  (A^T y = dL/dx with y = W z)
    build_rhs(g, dL_dU, nullptr, nullptr, false, g->bvec);
    int st = solve_system(g, g->bvec, g->xvec, true, info);
    const double* z = g->xvec;
    const double* zl = z + g->nfl;
    const double* zU = zl + 3 * (i64)g->nbl;
    const double* lam = x_fwd + g->nfl;
    const double* U = lam + 3 * (i64)g->nbl;
    if (dL_dslip && g->nbl) axpby<double>(dL_dslip, zl, -1.0, 0.0, 3 * (i64)g->nbl, g->s);
    if (dL_dr) adjoint_positions(g->d, g->nbl, g->bob, g->cur.r, x_fwd, lam, U, z, zl, zU, dL_dr, g->s);
    (void)n;
    ck(cudaStreamSynchronize(g->s));
    ck(cudaGetLastError());
    if (st) return fail(g, st, "mobility_solve_adjoint: adjoint solve did not converge");
  } catch (CudaError& e) {
    return fail(g, e.code, std::string("mobility_solve_adjoint: ") + e.what());
  }
  return RBFIB_OK;
}

}  // extern "C"

namespace {

// The body of one SEM step (Algorithm 1, steps 1-7).  Host-orchestrated
// (g->dev false): solves return their status and the rejection test is read
// on the host.  Captured for the device-driven step (g->dev true): the
// random-stream counters come from g->dstep, every solve is device-driven
// and the accept kernel copies the new configuration to (q, quat) unless a
// blob left the domain or a status word is set.  Returns the first nonzero
// solve status (host-orchestrated).
int sem_step_body(rbfib_grid* g, const rbfib_sem_params* p, uint64_t seed, uint64_t step, uint32_t attempt,
                  double* q, double* quat, rbfib_step_info& loc) {
  const int nb = g->nb, nbl = g->nbl;
  const double delta = p->delta > 0 ? p->delta : kDeltaDefault;
  const bool dev = g->dev;
  int st = 0;
  const i64 n = g->n_total();
  const cudaStream_t s = g->s;
  auto normals = [&](unsigned purpose, i64 count, double* out) {
    if (dev) philox_normals_p(g->dstep, purpose, count, out, g->s);
    else philox_normals(seed, step, attempt, purpose, count, out, g->s);
  };
  if (dev) ck(cudaMemsetAsync(g->dinfo.p, 0, sizeof(int) * 32, s));
  // current configuration
  if (nb) {
    ck(cudaMemcpyAsync(g->cur.q, q, sizeof(double) * 3 * nb, cudaMemcpyDeviceToDevice, s));
    ck(cudaMemcpyAsync(g->cur.quat, quat, sizeof(double) * 4 * nb, cudaMemcpyDeviceToDevice, s));
  }
  refresh_config(g, g->cur, true);
  // forces F^n
  body_forces(g->d, potentials_of(p), view_of(g, g->cur), p->force_ext, g->bodyF, s);
  if (p->no_rfd) {
    // naive Euler-Maruyama: no drift terms, step 6 only
    if (p->slip) ck(cudaMemcpyAsync(g->blobS, p->slip, sizeof(double) * 3 * nbl, cudaMemcpyDeviceToDevice, s));
    else ck(cudaMemsetAsync(g->blobS, 0, sizeof(double) * 3 * std::max(nbl, 1), s));
  } else {
    // step 1: random forces and torques W^FT = kT [W^f / L_p ; W^tau]
    normals(2u, 6 * (i64)nb, g->bodyWn);
    wft(nb, g->bodyWn, g->Lp, p->kT, g->bodyW, s);
    // step 2: constrained solve with W^FT (homogeneous)
    build_rhs(g, g->bodyW, nullptr, nullptr, false, g->bvec);
    int st1 = solve_system(g, g->bvec, g->xvec, true, &loc.solve_rfd, 0);
    if (st1) st = st1;
    ck(cudaMemcpyAsync(g->xrfd, g->xvec, sizeof(double) * n, cudaMemcpyDeviceToDevice, s));
    const double* v_rfd = g->xrfd;
    const double* lam_rfd = g->xrfd.p + g->nfl;
    const double* U_rfd = lam_rfd + 3 * (i64)nbl;
    // step 3: displaced configurations Q+- (lab-frame rotations by +-(delta/2) W^tau)
    move_bodies(nb, g->cur.q, g->cur.quat, g->bodyWn, g->Lp, 0.5 * delta, g->plus.q, g->plus.quat, s);
    move_bodies(nb, g->cur.q, g->cur.quat, g->bodyWn, g->Lp, -0.5 * delta, g->minus.q, g->minus.quat, s);
    refresh_config(g, g->plus, false);
    refresh_config(g, g->minus, false);
    // step 4: unconstrained Stokes solve with (S(Q+) - S(Q-)) lambda / delta
    ck(cudaMemsetAsync(g->bvec, 0, sizeof(double) * g->nfl, s));
    spread_diff(g->d, nbl, g->plus.r, g->minus.r, lam_rfd, 1.0 / (delta * g->dV), g->bvec, s);
    int st2 = solve_system(g, g->bvec, g->xvec, false, &loc.solve_stokes, 1);
    if (st2 && !st) st = st2;
    // step 5: random finite differences; F_tot = F - D^{K^T},
    // slip_tot = slip + D^K - D^J - D^S
    rfd_force(nb, g->boff, g->plus.arm, g->minus.arm, lam_rfd, 1.0 / delta, g->bodyF, s);
    rfd_slip(g->d, view_of(g, g->cur), g->plus.r, g->minus.r, g->plus.arm, g->minus.arm, v_rfd, U_rfd, g->xvec, p->slip,
             1.0 / delta, g->blobS, s);
  }
  // step 6: fluctuating constrained solve
  normals(1u, g->stress.total, g->Wst);
  stress_divergence(g->d, g->stress, g->Wst, std::sqrt(2.0 * g->desc.eta * p->kT / (g->dV * p->dt)), g->fnoise, s);
  build_rhs(g, g->bodyF, g->blobS, g->fnoise, true, g->bvec);
  int st3 = solve_system(g, g->bvec, g->xvec, true, &loc.solve_main, 2);
  if (st3 && !st) st = st3;
  // step 7: update and rejection test
  const double* Un = g->xvec.p + g->nfl + 3 * (i64)nbl;
  move_bodies(nb, g->cur.q, g->cur.quat, Un, nullptr, p->dt, g->next.q, g->next.quat, s);
  refresh_config(g, g->next, false);
  if (dev) {
    int* flag = g->dinfo.p + 12;
    outside_check(g->d, nbl, g->next.r, flag, s);
    accept_step(nb, flag, g->dinfo.p + 1, 4, 4, g->next.q, g->next.quat, q, quat, g->dinfo.p + 14, s);
    return 0;
  }
  int* flag = (int*)g->part.p;   // scratch word
  ck(cudaMemsetAsync(flag, 0, sizeof(int), s));
  outside_check(g->d, nbl, g->next.r, flag, s);
  int hflag = 0;
  ck(cudaMemcpyAsync(&hflag, flag, sizeof(int), cudaMemcpyDeviceToHost, s));
  ck(cudaStreamSynchronize(s));
  loc.rejected = hflag ? 1 : 0;
  if (!hflag && !st && nb) {
    ck(cudaMemcpyAsync(q, g->next.q, sizeof(double) * 3 * nb, cudaMemcpyDeviceToDevice, s));
    ck(cudaMemcpyAsync(quat, g->next.quat, sizeof(double) * 4 * nb, cudaMemcpyDeviceToDevice, s));
  }
  ck(cudaStreamSynchronize(s));
  ck(cudaGetLastError());
  return st;
}

// Whether the step graph can be used: a coupled body block needs a valid
// inverse at known orientations to warm-start from.
bool step_graph_ok(rbfib_grid* g) {
  return g->use_graphs && g->timer_kind == 0 && (!g->dense_body || (g->dM_valid && g->dquat_valid));
}

// Captures the device-driven step for (p, q, quat).  Returns false when the
// capture or instantiation failed (the host-orchestrated step is used then).
bool build_step_graph(rbfib_grid* g, const rbfib_sem_params* p, double* q, double* quat) {
  if (g->sgraph.exec) cudaGraphExecDestroy(g->sgraph.exec);
  g->sgraph = rbfib_grid::StepGraph();
  cudaStream_t s0 = g->s;
  const long long l0 = rbfib::g_launches.load();
  cudaGraph_t graph = nullptr;
  bool ok = true;
  g->dev = true;
  g->cap_depth = 0;
  g->cap_bodies = 0;
  g->s = cap_stream(g, 0);
  try {
    ck(cudaStreamBeginCapture(g->s, cudaStreamCaptureModeRelaxed));
    rbfib_step_info loc{};
    sem_step_body(g, p, 0, 0, 0, q, quat, loc);
    ck(cudaStreamEndCapture(g->s, &graph));
    ck(cudaGraphInstantiate(&g->sgraph.exec, graph, 0));
  } catch (CudaError&) {
    ok = false;
    cudaStreamCaptureStatus cst;
    if (cudaStreamIsCapturing(g->s, &cst) == cudaSuccess && cst != cudaStreamCaptureStatusNone) {
      cudaGraph_t t = nullptr;
      cudaStreamEndCapture(g->s, &t);
      if (t) cudaGraphDestroy(t);
    }
    cudaGetLastError();
  }
  if (graph) cudaGraphDestroy(graph);
  g->dev = false;
  g->cap_depth = 0;
  g->s = s0;
  const long long captured = (long long)rbfib::g_launches.load() - l0;
  g->cap_outside = captured - g->cap_bodies;
  rbfib::g_launches.fetch_sub((unsigned long long)captured);   // captured, not launched
  if (!ok) {
    g->sgraph = rbfib_grid::StepGraph();
    return false;
  }
  g->sgraph.q = q;
  g->sgraph.quat = quat;
  g->sgraph.p = *p;
  return true;
}

bool same_params(const rbfib_sem_params& a, const rbfib_sem_params& b) {
  return std::memcmp(&a, &b, sizeof(rbfib_sem_params)) == 0;
}

// Launches the device-driven step on g->s (no host synchronisation).
// Returns false if it could not be built (use the host-orchestrated step).
bool step_graph_launch(rbfib_grid* g, const rbfib_sem_params* p, uint64_t seed, uint64_t step, uint32_t attempt,
                       double* q, double* quat) {
  if (!step_graph_ok(g)) return false;
  if (!g->sgraph.exec || g->sgraph.q != q || g->sgraph.quat != quat || !same_params(g->sgraph.p, *p))
    if (!build_step_graph(g, p, q, quat)) { g->use_graphs = false; return false; }
  unsigned long long* hs = (unsigned long long*)(g->h_pinned + 48);
  hs[0] = seed; hs[1] = step; hs[2] = attempt;
  ck(cudaMemcpyAsync(g->dstep.p, hs, sizeof(unsigned long long) * 3, cudaMemcpyHostToDevice, g->s));
  ck(cudaGraphLaunch(g->sgraph.exec, g->s));
  int* hi = (int*)(g->h_pinned + 24);     // 32 ints: h_pinned[24..39]
  ck(cudaMemcpyAsync(hi, g->dinfo.p, sizeof(int) * 32, cudaMemcpyDeviceToHost, g->s));
  ck(cudaMemcpyAsync(g->h_pinned + 52, g->drel.p, sizeof(double) * 4, cudaMemcpyDeviceToHost, g->s));
  ck(cudaMemcpyAsync(g->h_pinned + 56, g->dwarm.p, sizeof(long long), cudaMemcpyDeviceToHost, g->s));
  return true;
}

// After the stream has been synchronised: the step's information and status.
int step_graph_finish(rbfib_grid* g, rbfib_step_info* info) {
  const int* hi = (const int*)(g->h_pinned + 24);
  const double* hr = g->h_pinned + 52;
  rbfib_step_info loc{};
  rbfib_solve_info* si[3] = {&loc.solve_rfd, &loc.solve_stokes, &loc.solve_main};
  int st = 0;
  long long launches = g->cap_outside;
  for (int k = 0; k < 3; ++k) {
    si[k]->iterations = hi[4 * k];
    si[k]->refinements = g->desc.precision == RBFIB_FP64 ? 0 : hi[4 * k + 2];
    si[k]->rel_residual = hr[k];
    if (hi[4 * k + 1] && !st) st = hi[4 * k + 1];
    g->gs_iters += hi[4 * k];
    g->reorth_passes += hi[4 * k + 3];
    // launches that ran: per pass of the WHILE body its fixed part, per
    // iteration its launches without the gated second pass, two per second
    // pass taken
    launches += (long long)hi[4 * k + 2] * g->cap_body_fixed[k] + (long long)hi[4 * k] * (g->cap_per_iter[k] - 2) +
                2LL * hi[4 * k + 3];
  }
  rbfib::g_launches.fetch_add((unsigned long long)std::max(launches, 0LL));
  g->ns_warm_dev = *(const long long*)(g->h_pinned + 56);
  loc.rejected = hi[14];
  if (info) *info = loc;
  if (hi[13]) {
    g->dM_valid = false;
    g->dquat_valid = false;
    drop_graphs(g);
    return fail(g, RBFIB_EINTERNAL, "sem_step: body block: zero pivot in the Gauss-Jordan inversion");
  }
  if (st) return fail(g, st, "sem_step: a solve did not converge");
  if (loc.rejected) return fail(g, RBFIB_EREJECT, "sem_step: unphysical configuration rejected");
  return RBFIB_OK;
}

}  // namespace

// Device-driven steps of ensemble systems (batch.cu).
bool rbfib_grid_step_launch(rbfib_grid* g, const rbfib_sem_params* p, uint64_t seed, uint64_t step,
                            uint32_t attempt, double* q, double* quat) {
  if (!g || !p || (g->nb > 0 && (!q || !quat)) || !(p->dt > 0) || !(p->kT >= 0) || !g->step_graphs ||
      (p->no_rfd != 0 && p->no_rfd != 1) || p->reserved != 0)
    return false;
  try {
    g->last_step_dev = step_graph_launch(g, p, seed, step, attempt, q, quat) ? 1 : 0;
    return g->last_step_dev != 0;
  } catch (CudaError&) {
    cudaGetLastError();
    return false;
  }
}

// Whether a grid's device-driven step can be captured now for these
// arguments (the checks of rbfib_grid_step_launch, and a valid body block).
bool rbfib_grid_step_ready(rbfib_grid* g, const rbfib_sem_params* p, const double* q, const double* quat) {
  return g && p && !(g->nb > 0 && (!q || !quat)) && p->dt > 0 && p->kT >= 0 && g->step_graphs &&
         (p->no_rfd == 0 || p->no_rfd == 1) && p->reserved == 0 && step_graph_ok(g);
}

// Puts a step's random-stream counters in the grid's pinned buffer, from
// which the batch graph's first node for this grid copies them.
void rbfib_grid_stage_step(rbfib_grid* g, uint64_t seed, uint64_t step, uint32_t attempt) {
  unsigned long long* hs = (unsigned long long*)(g->h_pinned + 48);
  hs[0] = seed; hs[1] = step; hs[2] = attempt;
  g->last_step_dev = 1;
}

// Captures the device-driven SEM steps of grids gs[0..n) as n parallel
// branches of one graph, instantiated into *out: each branch copies its
// grid's staged counters to the device, runs the step (restart cycles,
// refinement sweeps and the body block's warm start in the grid's own
// conditional nodes) and copies the step's report back to the grid's pinned
// buffer, as step_graph_launch does for one grid.  s is the stream the
// capture starts on (and the graph is launched on).  Returns false, with
// nothing captured left behind, when a grid is not ready or the capture or
// instantiation fails.
bool rbfib_batch_graph_build(rbfib_grid* const* gs, int n, const rbfib_sem_params* params, double* const* q,
                             double* const* quat, cudaStream_t s, cudaGraphExec_t* out) {
  *out = nullptr;
  for (int i = 0; i < n; ++i)
    if (!rbfib_grid_step_ready(gs[i], &params[i], q[i], quat[i])) return false;
  cudaGraph_t graph = nullptr;
  cudaEvent_t fork = nullptr;
  std::vector<cudaEvent_t> joins(n, nullptr);
  std::vector<cudaStream_t> saved(n, nullptr);
  for (int i = 0; i < n; ++i) saved[i] = gs[i]->s;
  bool ok = true;
  try {
    ck(cudaEventCreateWithFlags(&fork, cudaEventDisableTiming));
    for (int i = 0; i < n; ++i) ck(cudaEventCreateWithFlags(&joins[i], cudaEventDisableTiming));
    ck(cudaStreamBeginCapture(s, cudaStreamCaptureModeRelaxed));
    ck(cudaEventRecord(fork, s));
    for (int i = 0; i < n; ++i) {
      rbfib_grid* g = gs[i];
      const long long l0 = rbfib::g_launches.load();
      g->dev = true;
      g->cap_depth = 0;
      g->cap_bodies = 0;
      g->s = cap_stream(g, 0);
      ck(cudaStreamWaitEvent(g->s, fork, 0));
      ck(cudaMemcpyAsync(g->dstep.p, g->h_pinned + 48, sizeof(unsigned long long) * 3, cudaMemcpyHostToDevice,
                         g->s));
      rbfib_step_info loc{};
      sem_step_body(g, &params[i], 0, 0, 0, q[i], quat[i], loc);
      ck(cudaMemcpyAsync(g->h_pinned + 24, g->dinfo.p, sizeof(int) * 32, cudaMemcpyDeviceToHost, g->s));
      ck(cudaMemcpyAsync(g->h_pinned + 52, g->drel.p, sizeof(double) * 4, cudaMemcpyDeviceToHost, g->s));
      ck(cudaMemcpyAsync(g->h_pinned + 56, g->dwarm.p, sizeof(long long), cudaMemcpyDeviceToHost, g->s));
      ck(cudaEventRecord(joins[i], g->s));
      ck(cudaStreamWaitEvent(s, joins[i], 0));
      const long long captured = (long long)rbfib::g_launches.load() - l0;
      g->cap_outside = captured - g->cap_bodies;
      rbfib::g_launches.fetch_sub((unsigned long long)captured);   // captured, not launched
      g->dev = false;
      g->cap_depth = 0;
      g->s = saved[i];
    }
    ck(cudaStreamEndCapture(s, &graph));
    ck(cudaGraphInstantiate(out, graph, 0));
  } catch (CudaError&) {
    ok = false;
    // end the capture on the origin stream, then on any grid's capture
    // stream that a failure left joined to it, so every stream is usable
    auto end_capture = [](cudaStream_t st) {
      cudaStreamCaptureStatus cst;
      if (st && cudaStreamIsCapturing(st, &cst) == cudaSuccess && cst != cudaStreamCaptureStatusNone) {
        cudaGraph_t t = nullptr;
        cudaStreamEndCapture(st, &t);
        if (t) cudaGraphDestroy(t);
      }
    };
    end_capture(s);
    for (int i = 0; i < n; ++i) end_capture(gs[i]->cap_streams[0]);
    cudaGetLastError();
    if (*out) cudaGraphExecDestroy(*out);
    *out = nullptr;
  }
  for (int i = 0; i < n; ++i) {
    gs[i]->dev = false;
    gs[i]->cap_depth = 0;
    gs[i]->s = saved[i];
  }
  if (graph) cudaGraphDestroy(graph);
  if (fork) cudaEventDestroy(fork);
  for (cudaEvent_t e : joins)
    if (e) cudaEventDestroy(e);
  return ok;
}

int rbfib_grid_step_finish(rbfib_grid* g, rbfib_step_info* info) {
  try {
    ck(cudaGetLastError());
    return step_graph_finish(g, info);
  } catch (CudaError& e) {
    return fail(g, e.code, std::string("sem_step: ") + e.what());
  }
}

extern "C" {

// Algorithm 1 (Split-Euler-Maruyama), steps 1-7.  With graphs (the
// default) the whole step is one device-driven graph launch and one
// synchronisation; otherwise the host orchestrates it.
int rbfib_sem_step(rbfib_grid* g, const rbfib_sem_params* p, uint64_t seed, uint64_t step, uint32_t attempt,
                   double* q, double* quat, rbfib_step_info* info) {
  if (!g || !p || (g->nb > 0 && (!q || !quat)) || !(p->dt > 0) || !(p->kT >= 0) || (p->no_rfd != 0 && p->no_rfd != 1) ||
      p->reserved != 0)
    return fail(g, RBFIB_EINVAL, "sem_step: bad argument");
  rbfib_step_info loc{};
  int st = 0;
  try {
    if (g->step_graphs && step_graph_launch(g, p, seed, step, attempt, q, quat)) {
      g->last_step_dev = 1;
      ck(cudaStreamSynchronize(g->s));
      ck(cudaGetLastError());
      return step_graph_finish(g, info);
    }
    g->last_step_dev = 0;
    st = sem_step_body(g, p, seed, step, attempt, q, quat, loc);
  } catch (CudaError& e) {
    return fail(g, e.code, std::string("sem_step: ") + e.what());
  }
  if (info) *info = loc;
  if (st) return fail(g, st, "sem_step: a solve did not converge");
  if (loc.rejected) return fail(g, RBFIB_EREJECT, "sem_step: unphysical configuration rejected");
  return RBFIB_OK;
}

}  // extern "C"
