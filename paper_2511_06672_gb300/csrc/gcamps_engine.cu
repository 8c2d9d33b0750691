// Engine launch of libgcamps (arxiv 2511.06672, Sec. 3): the gate-list kernel k_run, the reset and
// the readout kernels (<W>, overlap).

#include "gcamps_device.cuh"

namespace gcx {
namespace {

__global__ void __launch_bounds__(kThreads, kMinCtas) k_run(Engine e, const gcamps_op* ops, const int32_t* begin) {
  const int c = blockIdx.x / e.csize;
  run_body(e, ops, begin[c], begin[c + 1], c, blockIdx.x % e.csize);
}


// |0...0> with C = I, counters cleared.
__global__ void __launch_bounds__(kThreads) k_reset(Engine e) {
  Ctx C = make_ctx(e, blockIdx.x);
  const int n = C.n, d = e.d;
  for (int i = threadIdx.x; i < 4 * n * n; i += blockDim.x) {
    const int row = i / (2 * n), col = i % (2 * n);
    // row j < n: Z_j -> z column n + j; row n + j: X_j -> x column j
    const uint8_t v = (row < n) ? (col == n + row) : (col == row - n);
    C.fx[i] = v;
    C.ix[i] = v;
  }
  for (int i = threadIdx.x; i < 2 * n; i += blockDim.x) {
    C.fr[i] = 0;
    C.ir[i] = 0;
    C.weyl[i] = 0;
  }
  for (int j = threadIdx.x; j < n; j += blockDim.x) {
    double2* A = site_ptr(C, j);
    for (int sidx = 0; sidx < d; ++sidx) A[sidx] = make_double2(sidx == 0 ? 1.0 : 0.0, 0.0);
  }
  for (int j = threadIdx.x; j <= n; j += blockDim.x) C.dims[j] = 1;
  if (threadIdx.x < M_COUNT) C.meta[threadIdx.x] = 0;
  if (threadIdx.x < S_COUNT) C.stats[threadIdx.x] = (threadIdx.x == S_MAXCHI) ? 1 : 0;
  if (C.prof && threadIdx.x < P_COUNT) C.prof[threadIdx.x] = 0;
  if (threadIdx.x < kDStats) C.dstats[threadIdx.x] = 0.0;
}

// ------------------------------------------------------------------------------ readouts
// <MPS| P' |MPS> with P' = C^dag W C = tau^r (x)_j X^{a_j} Z^{b_j}: the inverse-tableau rows are
// multiplied in the order of W = prod_j X_j^{x_j} Z_j^{z_j}, then transfer matrices left to right.

constexpr int kStage = 8192;    // entries of the staged state: 128 KB of dynamic shared memory
constexpr int kHalfE = 128;     // E's part of a half's share of s.z
__global__ void __launch_bounds__(kThreads) k_expect(Engine e, int c, const int8_t* xz, double2* out) {
  extern __shared__ __align__(16) double2 stage[];
  __shared__ Smem s;
  __shared__ int dim[kMaxN + 1], at[kMaxN + 1];
  __shared__ int acc_x[kMaxN], acc_z[kMaxN];
  __shared__ int acc_r;
  Ctx C = make_ctx(e, c);
  init_tau(s, e.d);
  const int n = C.n, d = e.d;
  conj_weyl(s, C, xz, acc_x, acc_z, &acc_r);
  for (int i = threadIdx.x; i < e.batch * M_COUNT; i += blockDim.x)   // the status words, for the host's one copy
    reinterpret_cast<int*>(out + 1)[i] = e.meta[i];
  // Where the sites' tensors fit shared memory (kStage entries in all; bonds up to 9 for 32 qutrits), they are staged
  // at once and the two halves of the chain are contracted at the same time, each by half the CTA with its E and T in
  // s.z; a chain of n dependent steps becomes n / 2, without a wait for global memory in any of them.
  for (int j = threadIdx.x; j <= n; j += blockDim.x) dim[j] = C.dims[j];
  __syncthreads();
  if (threadIdx.x < 32) {   // first entry of every site in the stage
    int base = 0;
    for (int j0 = 0; j0 < n; j0 += 32) {
      const int j = j0 + (int)threadIdx.x;
      const int mine = j < n ? dim[j] * d * dim[j + 1] : 0;
      int v = mine;
      for (int o = 1; o < 32; o <<= 1) {
        const int u = __shfl_up_sync(0xffffffffu, v, o);
        if ((int)threadIdx.x >= o) v += u;
      }
      if (j < n) at[j] = base + v - mine;
      base += __shfl_sync(0xffffffffu, v, 31);
      if (base > kStage) base = kStage + 1;   // too large: no overflow in what follows
    }
    if (threadIdx.x == 0) at[n] = base;
  }
  __syncthreads();
  bool ok = at[n] <= kStage;
  for (int j = threadIdx.x; j < n; j += blockDim.x)
    ok = ok && dim[j + 1] * dim[j + 1] <= kHalfE && dim[j] * d * dim[j + 1] <= kZ / 2 - kHalfE;
  if (__syncthreads_and(ok)) {
    for (int idx = threadIdx.x; idx < at[n]; idx += blockDim.x) {
      int lo = 0, hi = n;   // the site of entry idx
      while (hi - lo > 1) {
        const int mid = (lo + hi) / 2;
        if (at[mid] <= idx) lo = mid;
        else hi = mid;
      }
      stage[idx] = site_ptr(C, lo)[idx - at[lo]];
    }
    const int half = (int)threadIdx.x / (kThreads / 2);
    HalfGroup g{&s, (int)threadIdx.x % (kThreads / 2), kThreads / 2, half};
    double2* E = s.z + half * (kZ / 2);
    double2* T = E + kHalfE;
    if (g.tid == 0) E[0] = make_double2(1.0, 0.0);
    __syncthreads();
    const int mid = n / 2;
    if (half == 0)
      for (int j = 0; j < mid; ++j)
        transfer_site(g, s, E, T, stage + at[j], dim[j], dim[j + 1], stage + at[j], dim[j], dim[j + 1], d, acc_x[j],
                      acc_z[j]);
    else
      for (int j = n - 1; j >= mid; --j)
        transfer_site_left(g, s, E, T, stage + at[j], dim[j], dim[j + 1], d, acc_x[j], acc_z[j]);
    __syncthreads();
    if (threadIdx.x < 32) {
      double2 v = cz();
      for (int i = threadIdx.x; i < dim[mid] * dim[mid]; i += 32) v = cfma(s.z[i], s.z[kZ / 2 + i], v);
      v.x = warp_sum(v.x);
      v.y = warp_sum(v.y);
      if (threadIdx.x == 0) out[0] = cmul(s.tau[acc_r], v);
    }
    return;
  }
  double2* E = C.scr + e.sl.b;
  double2* T = C.scr + e.sl.tmp;
  if (threadIdx.x == 0) E[0] = make_double2(1.0, 0.0);
  __syncthreads();
  const BlockGroup g{&s, (int)threadIdx.x, (int)blockDim.x};
  for (int j = 0; j < n; ++j) {
    const double2* A = site_ptr(C, j);
    transfer_site(g, s, E, T, A, dim[j], dim[j + 1], A, dim[j], dim[j + 1], d, acc_x[j], acc_z[j]);
  }
  if (threadIdx.x == 0) out[0] = cmul(s.tau[acc_r], E[0]);
}

// <M1|M2> for circuit c1 of e1 and circuit c2 of e2 (same n and d; Sec. 2.4 MPS): transfer matrices
// E[a1][a2] from the left, T[a1][s][b2] = sum_a2 E[a1][a2] B[a2][s][b2], then
// E'[b1][b2] = sum_{a1, s} conj(A[a1][s][b1]) T[a1][s][b2]; FP64, one CTA, scratch of circuit c1.
__global__ void __launch_bounds__(kThreads) k_overlap(Engine e1, int c1, Engine e2, int c2, double2* out) {
  __shared__ Smem s;
  const Ctx A = make_ctx(e1, c1), B = make_ctx(e2, c2);
  const int n = A.n, d = e1.d;
  const bool fits = transfer_fits(A.dims, B.dims, n, d);
  double2* E = fits ? s.z : A.scr + e1.sl.b;
  double2* T = fits ? s.z + kTransferE : A.scr + e1.sl.tmp;
  if (threadIdx.x == 0) E[0] = make_double2(1.0, 0.0);
  __syncthreads();
  const BlockGroup g{&s, (int)threadIdx.x, (int)blockDim.x};
  for (int j = 0; j < n; ++j)
    transfer_site(g, s, E, T, site_ptr(A, j), A.dims[j], A.dims[j + 1], site_ptr(B, j), B.dims[j], B.dims[j + 1], d, 0, 0);
  if (threadIdx.x == 0) out[0] = E[0];
}

}  // namespace

cudaError_t launch_overlap(const Engine& e1, int c1, const Engine& e2, int c2, double2* out_dev, cudaStream_t st) {
  k_overlap<<<1, kThreads, 0, st>>>(e1, c1, e2, c2, out_dev);
  return cudaGetLastError();
}

cudaError_t launch_run(const Engine& e, const gcamps_op* ops_dev, const int32_t* begin_dev, cudaStream_t st) {
  if (e.precision) return launch_run_tc(e, ops_dev, begin_dev, st);
  return launch_cluster(k_run, e, st, e, ops_dev, begin_dev);
}

cudaError_t launch_reset(const Engine& e, cudaStream_t st) {
  k_reset<<<e.batch, kThreads, 0, st>>>(e);
  return cudaGetLastError();
}

cudaError_t launch_expect(const Engine& e, int circuit, const int8_t* xz_dev, double2* out_dev, cudaStream_t st) {
  constexpr int bytes = kStage * sizeof(double2);
  const cudaError_t a = cudaFuncSetAttribute(k_expect, cudaFuncAttributeMaxDynamicSharedMemorySize, bytes);
  if (a != cudaSuccess) return a;
  k_expect<<<1, kThreads, bytes, st>>>(e, circuit, xz_dev, out_dev);
  return cudaGetLastError();
}

}  // namespace gcx
