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

__global__ void __launch_bounds__(kThreads) k_expect(Engine e, int c, const int8_t* xz, double2* out) {
  __shared__ Smem s;
  __shared__ int acc_x[kMaxN], acc_z[kMaxN];
  __shared__ int acc_r;
  Ctx C = make_ctx(e, c);
  init_tau(s, e.d);
  const int n = C.n, d = e.d;
  conj_weyl(s, C, xz, acc_x, acc_z, &acc_r);
  // transfer matrices: E (chi x chi) starts as [[1]]
  const bool fits = transfer_fits(C.dims, C.dims, n, d);
  double2* E = fits ? s.z : C.scr + e.sl.b;
  double2* T = fits ? s.z + kTransferE : C.scr + e.sl.tmp;
  if (threadIdx.x == 0) E[0] = make_double2(1.0, 0.0);
  __syncthreads();
  for (int j = 0; j < n; ++j) {
    const int cl = C.dims[j], cr = C.dims[j + 1];
    const double2* A = site_ptr(C, j);
    const bool more = j + 1 < n;
    transfer_site(s, E, T, A, cl, cr, A, cl, cr, d, acc_x[j], acc_z[j], more ? site_ptr(C, j + 1) : nullptr,
                  more ? cr * d * C.dims[j + 2] : 0);
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
  for (int j = 0; j < n; ++j)
    transfer_site(s, E, T, site_ptr(A, j), A.dims[j], A.dims[j + 1], site_ptr(B, j), B.dims[j], B.dims[j + 1], d, 0, 0,
                  nullptr, 0);
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
  k_expect<<<1, kThreads, 0, st>>>(e, circuit, xz_dev, out_dev);
  return cudaGetLastError();
}

}  // namespace gcx
