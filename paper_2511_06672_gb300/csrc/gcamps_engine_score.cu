// Class scoring on a given two-site tensor (arxiv 2511.06672, Sec. 3): a CTA per class for tensors whose work fits
// shared memory, the engine's cluster kernel for larger ones, and the variant whose working memory is a static
// device array of the library (no allocation).

#include <algorithm>

#include "gcamps_device.cuh"

namespace gcx {
namespace {

// Scores of every class on a caller-provided theta (score_theta_body).
__global__ void __launch_bounds__(kThreads, kMinCtas) k_score_theta(Engine e, const double2* th, int cl, int cr,
                                                                   double* out_s2, double* out_vn, int* out_choice) {
  score_theta_body(e, th, cl, cr, out_s2, out_vn, out_choice);
}

// FP32 von Neumann estimates of every class on a caller-provided theta, with their error bounds (the pruning
// step of the disentangler, vn_est32), one class per CTA of the first circuit's cluster.
__global__ void __launch_bounds__(kThreads, kMinCtas) k_estimate_theta(Engine e, const double2* th, int cl, int cr,
                                                                      double* out_est, double* out_bd) {
  __shared__ Smem s;
  const int c = blockIdx.x / e.csize, rank = blockIdx.x % e.csize;
  if (c != 0) return;   // the whole cluster of every other circuit leaves together
  Ctx C = make_ctx(e, c, rank);
  const int d = C.d, dd = d * d;
  if (rank == 0)
    for (int i = threadIdx.x; i < cl * dd * cr; i += blockDim.x) C.th32[i] = make_float2((float)th[i].x, (float)th[i].y);
  cluster_sync();
  float2* ws = reinterpret_cast<float2*>(C.cta + e.cl.block);
  const int rows = cl * d, cols = d * cr;
  const double bound = vn_est_bound(d, rows < cols ? rows : cols, rows < cols ? cols : rows);
  for (int k = rank; k < C.K; k += C.csize) {
    float est = 0.f;
    BlockGroup g{&s, (int)threadIdx.x, (int)blockDim.x};
    const bool ok = vn_est32(g, C, C.th32, cl, cr, e.candU32 + (long long)k * dd * dd, ws, s.hv, s.hw, kBTri,
                             s.btri32, kBTri, &est, (float*)nullptr, (float*)nullptr);
    if (threadIdx.x == 0) {
      out_est[k] = est;
      out_bd[k] = ok ? bound : 1e300;
    }
    __syncthreads();
  }
  cluster_sync();
}

// theta' = Q theta and its Gram, `width` columns of the long side at a time: x holds the short side's m entries of each
// (short index major, padded stride, where the rows are short; long index major where the columns are).
template <class Grp>
__device__ void gram_chunked(const Grp& g, const double2* theta, int cl, int cr, int d, const double2* Q, double2* G,
                             double2* x, int width) {
  const int dd = d * d, rows = cl * d, cols = d * cr;
  const bool wide = rows <= cols;
  const int m = wide ? rows : cols, M = wide ? cols : rows, ntri = m * (m + 1) / 2;
  const int ld = wide ? (width | 1) : m;
  for (int c0 = 0; c0 < M; c0 += width) {
    const int w = min(width, M - c0);
    for (int idx = g.tid; idx < m * w; idx += g.n) {
      const int i = wide ? idx / w : idx % m, c = wide ? idx % w : idx / m;
      const int rr = wide ? i : c0 + c, col = wide ? c0 + c : i;
      const int a = rr / d, sd = rr % d, t = col / cr, b = col % cr;
      const double2* q = Q + (sd * d + t) * dd;
      const double2* th = theta + (long long)a * dd * cr + b;
      double2 acc = cz();
      for (int u = 0; u < dd; ++u) acc = cfma(q[u], th[(long long)u * cr], acc);
      x[wide ? i * ld + c : c * ld + i] = acc;
    }
    g.sync();
    for (int idx = g.tid; idx < ntri; idx += g.n) {
      int i, j;
      tri_index(idx, i, j);
      double2 acc = c0 ? G[i * m + j] : cz();
      if (wide)
        for (int c = 0; c < w; ++c) acc = cfmac(x[j * ld + c], x[i * ld + c], acc);   // sum_c x_i conj(x_j)
      else
        for (int c = 0; c < w; ++c) acc = cfmac(x[c * ld + i], x[c * ld + j], acc);
      G[i * m + j] = acc;
      if (c0 + width >= M && i != j) G[j * m + i] = cconj(acc);
    }
    g.sync();
  }
}

// Every class of one theta at once: CTA k < K takes the exact FP64 scores of class k, CTA K + k its FP32 screen and
// estimate, into rows of kMaxK doubles (KnownScore).  The classes are independent, and 90 CTAs on 152 SMs take the
// time of one: 1.6 ms at m = 75 instead of 42 for the classes in turn on a cluster of 4.  theta', the Gram and the
// reduction's scratch live in dynamic shared memory (kGridMax entries of theta).  Below kGridWarpM rows a CTA is one
// warp (the steps of a reduction of so few rows fit one).
constexpr int kGridMax = 81 * 81, kGridWarpM = 10, kGridWidth = 32;
template <class Grp>
__device__ __forceinline__ void score_grid_body(Smem& s, const Grp& g, const Engine& e, const double2* th, int cl,
                                                int cr, double* out) {
  extern __shared__ __align__(16) unsigned char dyn[];
  Ctx C = {};
  C.e = &e;
  C.d = e.d;
  C.K = e.K;
  C.rank = 1;   // not a leader: no counters
  const int d = e.d, dd = d * d, rows = cl * d, cols = d * cr;
  const int m = min(rows, cols), M = max(rows, cols);
  const int k = blockIdx.x % e.K;
  constexpr bool kWarpLevel = Grp::kSize == 32;
  if (blockIdx.x < e.K) {
    double2* G = reinterpret_cast<double2*>(dyn);
    double* dg = reinterpret_cast<double*>(G + m * m);
    double* od = dg + m;
    gram_chunked(g, th, cl, cr, d, e.candU + (long long)k * dd * dd, G, G + m * m + m, min(M, kGridWidth));
    double tr = 0, fro = 0;
    for (int idx = g.tid; idx < m * m; idx += g.n) {
      const double2 v = G[idx];
      if (idx / m == idx % m) tr += v.x;
      fro += cabs2(v);
    }
    tr = g.sum(tr);
    fro = g.sum(fro);
    const Score sc = score_spectrum(g, C, G, m, tr, fro, true, dg, od, kWarpLevel ? s.wtri[0] : s.btri,
                                    kWarpLevel ? s.wtri32[0] : s.btri32, kWarpLevel ? 32 : kBTri);
    if (g.tid == 0) {
      out[kKnownS2 * kMaxK + k] = sc.s2;
      out[kKnownVn * kMaxK + k] = sc.vn;
      out[kKnownRank * kMaxK + k] = sc.rank;
    }
  } else {
    float2* th32 = reinterpret_cast<float2*>(dyn);
    for (int i = g.tid; i < rows * cols; i += g.n) th32[i] = make_float2((float)th[i].x, (float)th[i].y);
    g.sync();
    float est = 0.f, v = 0.f, lo = 0.f;
    const bool ok = vn_est32(g, C, th32, cl, cr, e.candU32 + (long long)k * dd * dd, th32 + rows * cols,
                             kWarpLevel ? s.whv[0] : s.hv, kWarpLevel ? s.whw[0] : s.hw, kWarpLevel ? 32 : kBTri,
                             kWarpLevel ? s.wtri32[0] : s.btri32, kWarpLevel ? 32 : kBTri, &est, &v, &lo);
    if (g.tid == 0) {
      out[kKnownScreen * kMaxK + k] = v;
      out[kKnownScreenLo * kMaxK + k] = lo;
      out[kKnownEst * kMaxK + k] = est;
      out[kKnownBound * kMaxK + k] = ok ? vn_est_bound(d, m, M) : 1e300;
    }
  }
}
struct GridWarp : WarpGroup {
  static constexpr int kSize = 32;
};
struct GridBlock : BlockGroup {
  static constexpr int kSize = kThreads;
};
__global__ void __launch_bounds__(32) k_score_grid_warp(Engine e, const double2* th, int cl, int cr, double* out) {
  __shared__ Smem s;
  GridWarp g;
  g.tid = (int)threadIdx.x;
  score_grid_body(s, g, e, th, cl, cr, out);
}
__global__ void __launch_bounds__(kThreads, 1) k_score_grid(Engine e, const double2* th, int cl, int cr, double* out) {
  __shared__ Smem s;
  GridBlock g;
  g.s = &s;
  g.tid = (int)threadIdx.x;
  g.n = (int)blockDim.x;
  score_grid_body(s, g, e, th, cl, cr, out);
}

// The disentangler's choice from the scores of k_score_grid, through select_class (e.csize as its cluster size); the
// scores go to the caller's arrays.  choice: class, exact evaluations that the bounds leave, and (status) the device
// status.
__global__ void __launch_bounds__(kThreads) k_score_choice(Engine e, const double2* th, int cl, int cr,
                                                           const double* known, double* out_s2, double* out_vn,
                                                           int* out_choice, bool status) {
  __shared__ Smem s;
  Ctx C = {};
  C.e = &e;
  C.csize = e.csize;
  C.d = e.d;
  C.K = e.K;
  C.known = known;
  for (int k = threadIdx.x; k < C.K; k += blockDim.x) {
    out_s2[k] = known[kKnownS2 * kMaxK + k];
    out_vn[k] = known[kKnownVn * kMaxK + k];
  }
  score_classes(s, &s, C, th, cl, cr, nullptr, C.K, kExact);
  __syncthreads();
  int nev = 0;
  const int kb = select_class(s, &s, C, th, cl, cr, &nev, false);
  if (threadIdx.x == 0) {
    out_choice[0] = kb;
    out_choice[1] = nev;
    if (status) out_choice[2] = 0;   // no iteration of the scoring can fail
  }
}

// Dynamic shared memory of the scores of a theta with sides m <= M: the exact ones' (Gram, tridiagonal, a chunk of
// theta'), the estimates' (theta, theta' and the Gram in FP32, three arrays of m).
constexpr size_t grid_bytes(int m, int M) {
  const size_t exact = (size_t)(m * m + m + m * ((M < kGridWidth ? M : kGridWidth) | 1)) * sizeof(double2);
  const size_t est = (size_t)(2 * m * M + m * m + 3 * m) * sizeof(float2);
  return exact > est ? exact : est;
}
// The most that any theta needs: m M <= kGridMax and m <= M, so no term is larger than at m = M = 81.
constexpr int kGridSide = 81;
constexpr size_t kGridBytes = grid_bytes(kGridSide, kGridSide);
static_assert(kGridSide * kGridSide == kGridMax && kGridBytes + sizeof(Smem) <= 227 * 1024, "fits a CTA");

// k_score_grid and k_score_choice for a theta of at most kGridMax entries; known: kKnownRows kMaxK doubles.
cudaError_t launch_grid(const Engine& e, const double2* th, int cl, int cr, double* known, double* s2, double* vn,
                        int* choice, bool status, cudaStream_t st) {
  const int rows = cl * e.d, cols = e.d * cr, m = std::min(rows, cols), M = std::max(rows, cols);
  const size_t bytes = grid_bytes(m, M);
  const bool warp = m < kGridWarpM;
  auto kern = warp ? k_score_grid_warp : k_score_grid;
  // more than a kernel gets unasked: the limit belongs to the kernel, not to the launch, so every call sets the same
  // one (with its own size a call on another thread could lower it between this one's set and its launch)
  if (bytes + sizeof(Smem) > 48 * 1024) {
    const cudaError_t a = cudaFuncSetAttribute(kern, cudaFuncAttributeMaxDynamicSharedMemorySize, (int)kGridBytes);
    if (a != cudaSuccess) return a;
  }
  kern<<<2 * e.K, warp ? 32 : kThreads, bytes, st>>>(e, th, cl, cr, known);
  cudaError_t ce = cudaGetLastError();
  if (ce != cudaSuccess) return ce;
  k_score_choice<<<1, kThreads, 0, st>>>(e, th, cl, cr, known, s2, vn, choice, status);
  return cudaGetLastError();
}

}  // namespace

cudaError_t launch_estimate_theta(const Engine& e, const double2* th, int cl, int cr, double* est, double* bd,
                                  cudaStream_t st) {
  return launch_cluster(k_estimate_theta, e, st, e, th, cl, cr, est, bd);
}

cudaError_t launch_score_theta(const Engine& e, const double2* th, int cl, int cr, double* s2, double* vn,
                               int* choice, double* known, cudaStream_t st) {
  if (e.precision) return launch_score_theta_tc(e, th, cl, cr, s2, vn, choice, st);
  if ((long long)cl * e.d * e.d * cr <= kGridMax) return launch_grid(e, th, cl, cr, known, s2, vn, choice, false, st);
  return launch_cluster(k_score_theta, e, st, e, th, cl, cr, s2, vn, choice);
}

// ------------------------------------------------------ class scores without device allocation
// gcamps_score_theta_noalloc: the scores of every class and the choice's record in the static array below (the rest
// of the work is in shared memory).
constexpr long long kStaticScores = (3LL * kMaxK + 2 + 2LL * kSmall + 15) / 16 * 16;
constexpr long long kStaticKnown = ((long long)kKnownRows * kMaxK + 15) / 16 * 16;
constexpr long long kStaticWords = kStaticScores + kStaticKnown;
static_assert(kStaticWords * 8 == 19072, "scratch size stated in gcamps.h");
static_assert(kStaticSide * kStaticSide <= kGridMax, "every accepted tensor takes the grid");
// Held by every device that loads the library.  Calls reuse it and it keeps the last call's contents, which no
// later call reads.
static __device__ __align__(256) double g_static_scratch[kStaticWords];
// Class unitaries for d = 2 then d = 3 ([K][d^4]) and their images ([K][20]), set once per device.
static __device__ __align__(256) double2 g_static_candU[kStaticK2 * 16 + kStaticK3 * 81];
static __device__ __align__(256) float2 g_static_candU32[kStaticK2 * 16 + kStaticK3 * 81];
static __device__ __align__(256) int32_t g_static_candImg[(kStaticK2 + kStaticK3) * 20];

// Device addresses of the arrays above, per device (host code only sees host-side stand-ins under
// their names).
struct StaticPtrs {
  double* scratch;
  double2* candU;
  float2* candU32;
  int32_t* candImg;
};
static StaticPtrs g_static_ptrs[kStaticMaxDevices];

cudaError_t static_setup(int device, const double* u2, const int32_t* img2, const double* u3,
                         const int32_t* img3) {
  if (device < 0 || device >= kStaticMaxDevices) return cudaErrorInvalidDevice;
  StaticPtrs p = {};
  cudaError_t ce = cudaGetSymbolAddress(reinterpret_cast<void**>(&p.scratch), g_static_scratch);
  if (ce == cudaSuccess) ce = cudaGetSymbolAddress(reinterpret_cast<void**>(&p.candU), g_static_candU);
  if (ce == cudaSuccess) ce = cudaGetSymbolAddress(reinterpret_cast<void**>(&p.candU32), g_static_candU32);
  if (ce == cudaSuccess) {
    float u32[2 * (kStaticK2 * 16 + kStaticK3 * 81)];
    for (int i = 0; i < 2 * kStaticK2 * 16; ++i) u32[i] = (float)u2[i];
    for (int i = 0; i < 2 * kStaticK3 * 81; ++i) u32[2 * kStaticK2 * 16 + i] = (float)u3[i];
    ce = cudaMemcpyToSymbol(g_static_candU32, u32, sizeof u32, 0);
  }
  if (ce == cudaSuccess) ce = cudaGetSymbolAddress(reinterpret_cast<void**>(&p.candImg), g_static_candImg);
  if (ce == cudaSuccess) ce = cudaMemcpyToSymbol(g_static_candU, u2, sizeof(double2) * kStaticK2 * 16, 0);
  if (ce == cudaSuccess)
    ce = cudaMemcpyToSymbol(g_static_candU, u3, sizeof(double2) * kStaticK3 * 81, sizeof(double2) * kStaticK2 * 16);
  if (ce == cudaSuccess) ce = cudaMemcpyToSymbol(g_static_candImg, img2, sizeof(int32_t) * kStaticK2 * 20, 0);
  if (ce == cudaSuccess)
    ce = cudaMemcpyToSymbol(g_static_candImg, img3, sizeof(int32_t) * kStaticK3 * 20, sizeof(int32_t) * kStaticK2 * 20);
  if (ce == cudaSuccess) g_static_ptrs[device] = p;
  return ce;
}

cudaError_t launch_score_theta_static(int device, int d, double tie_tol, const double2* th, int cl, int cr,
                                      double* s2, double* vn, int32_t* choice, cudaStream_t st) {
  if (device < 0 || device >= kStaticMaxDevices) return cudaErrorInvalidDevice;
  const StaticPtrs& p = g_static_ptrs[device];
  if (!p.scratch || !p.candU || !p.candU32 || !p.candImg) return cudaErrorInitializationError;
  Engine e = {};
  e.d = d;
  e.K = d == 2 ? kStaticK2 : kStaticK3;
  e.batch = 1;
  e.csize = kStaticCluster;
  e.tie_tol = tie_tol;
  e.lastsc = p.scratch;
  e.candU = p.candU + (d == 2 ? 0 : kStaticK2 * 16);
  e.candU32 = p.candU32 + (d == 2 ? 0 : kStaticK2 * 16);
  e.candImg = p.candImg + (d == 2 ? 0 : kStaticK2 * 20);
  return launch_grid(e, th, cl, cr, p.scratch + kStaticScores, s2, vn, choice, true, st);
}


}  // namespace gcx
