// Dense readout of libgcamps (arxiv 2511.06672, Sec. 3): psi = C|MPS> for small registers.
//
// C is written as a word of elementary Cliffords (found by elimination on the tableau, Sec. 2.2) and the word is
// applied to the dense MPS: a pass of d^n entries per Fourier gate, at most n^2 + 3 n of them (one for each site from j
// on in both reductions of each j, and two more), where summing C|x> over all x costs d^2n.  8 qutrits: 0.39 ms a call
// instead of 5.6, most of it launch and copy; 12 qutrits 17.6 ms instead of 1420, 20 qubits 55 instead of 5126 (on the 16
// SMs of the cluster at every size).

#include "gcamps_device.cuh"

namespace gcx {
namespace {

constexpr int kDenseN = 20;         // d^n <= 2^20
constexpr int kDenseGates = 1536;   // per site at most 2 (n - j) times three gates and four more
constexpr int kDenseCluster = 16;

// One gate: kind, site(s) and power packed in an int.  kSum: x_target += p x_control; kPhase: S^p; kFlip: |j> -> |-j>;
// kFourier: H^p (p = 1 or -1), the only one that is not monomial.
enum DenseKind { kPhase = 0, kSum = 1, kFlip = 2, kFourier = 3 };
__host__ __device__ constexpr int dense_gate(int kind, int q, int t, int p) { return kind | q << 4 | t << 12 | (p & 7) << 20; }

// The word of C: gates g_1 .. g_T with G = g_T .. g_1 and G C a Pauli string Q times a phase, Q = (x)_j X_j^{qx_j}
// Z_j^{qz_j}.  Row by row on a copy of the tableau: C X_j C^dag is turned into X_j (its other sites cleared with SUM
// from an X-only form), then C Z_j C^dag into Z_j with gates that keep X_j (in the frame after H on j).
struct DenseWord {
  uint8_t x[2 * kDenseN][kDenseN], z[2 * kDenseN][kDenseN];   // rows: Z_0.., X_0..
  int r[2 * kDenseN];
  int gates[kDenseGates];
  int count;
  int qx[kDenseN], qz[kDenseN];
};

// Conjugates every row by one gate and appends it.  Images: S: X -> tau^{[d = 2]} X Z; H: X -> Z, Z -> X^{-1};
// SUM: X_c -> X_c X_t, Z_t -> Z_t Z_c^{-1}; flip: X -> X^{-1}, Z -> Z^{-1}; rows are kept in the order X^x Z^z.
template <int D>
__device__ void dense_apply(DenseWord& w, int n, int kind, int q, int t, int p) {
  const int i = threadIdx.x;
  if (i < 2 * n) {
    int x = w.x[i][q], z = w.z[i][q];
    if (kind == kPhase) {
      w.r[i] = (w.r[i] + p * (x * (x - 1) + (D == 2 ? x : 0))) % (2 * D);
      z = (z + p * x) % D;
    } else if (kind == kFlip) {
      x = (D - x) % D;
      z = (D - z) % D;
    } else if (kind == kFourier) {
      const int x0 = x, z0 = z;
      w.r[i] = (w.r[i] + 2 * (D - (x0 * z0) % D)) % (2 * D);
      x = p > 0 ? (D - z0) % D : z0;
      z = p > 0 ? x0 : (D - x0) % D;
    } else {
      w.x[i][t] = (uint8_t)((w.x[i][t] + p * x) % D);
      z = (z + (D - p) * w.z[i][t]) % D;
    }
    w.x[i][q] = (uint8_t)x;
    w.z[i][q] = (uint8_t)z;
  }
  if (threadIdx.x == 0 && w.count < kDenseGates) w.gates[w.count++] = dense_gate(kind, q, t, p);
  __syncthreads();
}
// Makes row i X-only on the sites j.. and clears all of them but j (exponent a on X_j left); sites below j are 1.
template <int D>
__device__ void dense_reduce(DenseWord& w, int n, int i, int j) {
  for (int k = j; k < n; ++k) {
    const int x = w.x[i][k], z = w.z[i][k];
    __syncthreads();
    if (z == 0) continue;
    if (x == 0) dense_apply<D>(w, n, kFourier, k, k, 1);
    else dense_apply<D>(w, n, kPhase, k, k, (D - z) * x % D);   // 1 / x = x for x = 1, 2 mod 3
  }
  if (w.x[i][j] == 0) {
    int k = j + 1;
    while (k < n && w.x[i][k] == 0) ++k;
    __syncthreads();
    if (k < n) dense_apply<D>(w, n, kSum, k, j, 1);   // a row of a valid tableau has such a k
  }
  for (int k = j + 1; k < n; ++k) {
    const int a = w.x[i][j], b = w.x[i][k];
    __syncthreads();
    if (b) dense_apply<D>(w, n, kSum, j, k, (D - b) * a % D);
  }
}
template <int D>
__device__ void dense_word(DenseWord& w, const Ctx& C) {
  const int n = C.n;
  for (int idx = threadIdx.x; idx < 2 * n * n; idx += blockDim.x) {
    const int i = idx / n, j = idx % n;
    w.x[i][j] = C.fx[(long long)i * 2 * n + j];
    w.z[i][j] = C.fx[(long long)i * 2 * n + n + j];
  }
  for (int i = threadIdx.x; i < 2 * n; i += blockDim.x) w.r[i] = C.fr[i];
  if (threadIdx.x == 0) w.count = 0;
  __syncthreads();
  for (int j = 0; j < n; ++j) {
    dense_reduce<D>(w, n, n + j, j);
    const bool inverse = w.x[n + j][j] == 2;
    __syncthreads();
    if (inverse) dense_apply<D>(w, n, kFlip, j, j, 1);
    dense_apply<D>(w, n, kFourier, j, j, 1);     // X_j -> Z_j, Z_j X_j^b .. -> X_j^{-1} Z_j^b ..
    dense_reduce<D>(w, n, j, j);                 // S and SUM from j keep Z_j
    dense_apply<D>(w, n, kFourier, j, j, -1);
  }
  // G C: Z_j -> tau^r Z_j, X_j -> tau^r' X_j is conjugation by (x)_j X_j^{-r/2} Z_j^{r'/2}
  if ((int)threadIdx.x < n) {
    const int j = threadIdx.x;
    w.qx[j] = (D - (w.r[j] / 2) % D) % D;
    w.qz[j] = (w.r[n + j] / 2) % D;
  }
  __syncthreads();
}

// Digits of an index, two bits each, site 0 the most significant digit of the index and the lowest bits of the code.
template <int D>
__device__ __forceinline__ unsigned long long digits_of(int y, int n) {
  unsigned long long c = 0;
  for (int j = n - 1; j >= 0; --j) {
    c |= (unsigned long long)(y % D) << (2 * j);
    y /= D;
  }
  return c;
}
template <int D>
__device__ __forceinline__ int index_of(unsigned long long c, int n) {
  int y = 0;
  for (int j = 0; j < n; ++j) y = y * D + (int)((c >> (2 * j)) & 3);
  return y;
}

// Entry `code` of (gates[lo .. hi) in the word's order, inverted) applied to v: the inverses of monomial gates run in
// the order hi - 1 .. lo, so the output's source is found from lo up.  pauli: Q comes before them.
template <int D>
__device__ __forceinline__ double2 dense_entry(const DenseWord& w, const double2* v, const double2* tau, int n, int lo, int hi,
                                               bool pauli, unsigned long long code) {
  int ph = 0;
  for (int i = lo; i < hi; ++i) {
    const int g = w.gates[i], kind = g & 15, q = (g >> 4) & 255, t = (g >> 12) & 255, p = (g >> 20) & 7;
    const int jq = (int)(code >> (2 * q)) & 3;
    if (kind == kPhase) {   // S^{-p}: tau^{-p (j (j - 1) + [d = 2] j)}
      ph += (2 * D - 1) * p * (jq * (jq - 1) + (D == 2 ? jq : 0));
    } else {
      const int s = kind == kSum ? t : q, old = (int)(code >> (2 * s)) & 3;
      const int now = kind == kSum ? (old + p * jq) % D : (D - old) % D;   // SUM^{-p} |c, j> = |c, j - p c>
      code ^= (unsigned long long)(old ^ now) << (2 * s);
    }
  }
  if (pauli)
    for (int j = 0; j < n; ++j) {   // (X^a Z^b v)(y) = omega^{b (y - a)} v(y - a)
      const int old = (int)(code >> (2 * j)) & 3, now = (old + D - w.qx[j]) % D;
      code ^= (unsigned long long)(old ^ now) << (2 * j);
      ph += 2 * w.qz[j] * now;
    }
  const double2 x = __ldcg(v + index_of<D>(code, n));
  ph %= 2 * D;
  return ph ? cmul(tau[ph], x) : x;
}

// H^{-1} (sign > 0: the gate was H) or H on the d values u, without the factor d^{-1/2}.
template <int D>
__device__ __forceinline__ void small_fourier(double2* u, bool conj) {
  if (D == 2) {
    const double2 a = u[0], b = u[1];
    u[0] = cadd(a, b);
    u[1] = csub(a, b);
  } else {
    const double h = conj ? -0.86602540378443864676 : 0.86602540378443864676;   // Im omega^{+-1}
    const double2 a = u[0], t = cadd(u[1], u[2]), m = csub(u[1], u[2]);
    const double2 c = make_double2(fma(-0.5, t.x, a.x), fma(-0.5, t.y, a.y));
    u[0] = cadd(a, t);
    u[1] = make_double2(fma(-h, m.y, c.x), fma(h, m.x, c.y));
    u[2] = make_double2(fma(h, m.y, c.x), fma(-h, m.x, c.y));
  }
}

__device__ __forceinline__ unsigned long long mix64(unsigned long long z) {
  z += 0x9E3779B97F4A7C15ull;
  z = (z ^ (z >> 30)) * 0xBF58476D1CE4E5B9ull;
  z = (z ^ (z >> 27)) * 0x94D049BB133111EBull;
  return z ^ (z >> 31);
}

// psi(y) for the requested labels (all if ys is null), on one cluster, and behind them 1 if the state's bonds exceed their
// Schmidt bounds (nothing else is written then), else 0.  work: 4 dim entries, then one per CTA.  The
// phase of C is the one that gives C|0> = P v / |P v|, P the projector on the stabilizer rows' +1 eigenvector and v a
// fixed hashed vector: that of <C 0|v>, so |0> goes through the same passes.
template <int D>
__device__ void dense_body(DenseWord& w, Smem& s, const Engine& e, int c, int dim, const int32_t* ys, int nys, double2* work,
                           double2* out) {
  const Ctx C = make_ctx(e, c);
  const int n = C.n, rank = blockIdx.x, csize = gridDim.x;
  const int gt = rank * kThreads + threadIdx.x, gn = csize * kThreads;
  init_tau(s, D);
  double2* cur = work;
  double2* nxt = work + dim;
  double2* cur0 = work + 2LL * dim;
  double2* nxt0 = work + 3LL * dim;
  double2* part = work + 4LL * dim;
  dense_word<D>(w, C);   // every CTA: cheaper than sending it round
  // the dense MPS: d^{j+1} chi_{j+1} <= dim entries after site j, as every bond is within its Schmidt bound
  int rows = 1, chi = 1;
  bool fits = true;   // the same on every CTA
  for (int j = 0, r = D; j < n; ++j, r *= D) fits = fits && (long long)r * C.dims[j + 1] <= dim;
  // a state beyond them is none that this engine leaves: not read, and the caller is told by the entry behind the outputs
  if (gt == 0) out[nys] = make_double2(fits ? 0.0 : 1.0, 0.0);
  if (!fits) {
    cluster_sync();
    return;
  }
  for (int j = 0; j < n; ++j) {
    const int cr = C.dims[j + 1], wd = D * cr;
    const double2* A = site_ptr(C, j);
    for (int idx = gt; idx < rows * wd; idx += gn) {
      const int row = idx / wd, col = idx % wd;
      double2 acc = j ? cz() : A[col];
      if (j)
        for (int k = 0; k < chi; ++k) acc = cfma(__ldcg(cur + (long long)row * chi + k), A[(long long)k * wd + col], acc);
      __stcg(nxt + idx, acc);
    }
    cluster_sync();
    double2* t = cur;
    cur = nxt;
    nxt = t;
    rows *= D;
    chi = cr;
  }
  for (int y = gt; y < dim; y += gn) __stcg(cur0 + y, make_double2(y == 0 ? 1.0 : 0.0, 0.0));
  cluster_sync();
  // the word backwards, a pass per Fourier gate: the monomial gates found after it come first, read through
  int hi = w.count, nf = 0;
  bool pauli = true;
  while (true) {
    int f = hi - 1;
    while (f >= 0 && (w.gates[f] & 15) != kFourier) --f;
    const int q = f >= 0 ? (w.gates[f] >> 4) & 255 : 0;
    const bool conj = f >= 0 && ((w.gates[f] >> 20) & 7) == 1;   // undoing H: omega^{-ij}
    if (f >= 0) ++nf;
    int stride = 1;
    for (int j = q + 1; j < n; ++j) stride *= D;
    const int items = f >= 0 ? dim / D : dim;
    for (int idx = gt; idx < 2 * items; idx += gn) {
      const bool second = idx >= items;
      const int it = second ? idx - items : idx;
      const double2* src = second ? cur0 : cur;
      double2* dst = second ? nxt0 : nxt;
      if (f < 0) {
        __stcg(dst + it, dense_entry<D>(w, src, s.tau, n, 0, hi, pauli, digits_of<D>(it, n)));
        continue;
      }
      const int base = (it / stride) * stride * D + it % stride;
      const unsigned long long code = digits_of<D>(base, n);
      double2 u[D];
#pragma unroll
      for (int a = 0; a < D; ++a)
        u[a] = dense_entry<D>(w, src, s.tau, n, f + 1, hi, pauli, code | (unsigned long long)a << (2 * q));
      small_fourier<D>(u, conj);
#pragma unroll
      for (int a = 0; a < D; ++a) __stcg(dst + base + a * stride, u[a]);
    }
    cluster_sync();
    double2* t = cur;
    cur = nxt;
    nxt = t;
    t = cur0;
    cur0 = nxt0;
    nxt0 = t;
    pauli = false;
    if (f < 0) break;
    hi = f;
  }
  // <C 0|v>, a partial sum per CTA, added by every CTA in the same order
  double re = 0, im = 0;
  for (int y = gt; y < dim; y += gn) {
    const unsigned long long h = mix64((unsigned long long)y * 2 + 1), g = mix64((unsigned long long)y * 2 + 2);
    const double2 v = make_double2((double)(h >> 11) / 9007199254740992.0 - 0.5, (double)(g >> 11) / 9007199254740992.0 - 0.5);
    const double2 o = __ldcg(cur0 + y);
    re = fma(o.x, v.x, fma(o.y, v.y, re));
    im = fma(o.x, v.y, fma(-o.y, v.x, im));
  }
  re = block_sum(re, s);
  im = block_sum(im, s);
  if (threadIdx.x == 0) __stcg(part + rank, make_double2(re, im));
  cluster_sync();
  double2 tot = cz();
  for (int k = 0; k < csize; ++k) tot = cadd(tot, __ldcg(part + k));
  const double a2 = cabs2(tot);
  double scale = a2 > 0 ? 1.0 / sqrt(a2) : 0.0;
  for (int k = 0; k < nf / 2; ++k) scale /= D;   // nf factors d^{-1/2}
  if (nf & 1) scale /= sqrt((double)D);
  const double2 f = cscale(tot, scale);
  for (int t = gt; t < nys; t += gn) out[t] = cmul(f, __ldcg(cur + (ys ? ys[t] : t)));
  cluster_sync();
}

__global__ void __launch_bounds__(kThreads) k_dense(Engine e, int c, int dim, const int32_t* ys, int nys, double2* work,
                                                    double2* out) {
  __shared__ Smem s;
  __shared__ DenseWord w;
  if (e.d == 2) dense_body<2>(w, s, e, c, dim, ys, nys, work, out);
  else dense_body<3>(w, s, e, c, dim, ys, nys, work, out);
}

}  // namespace

size_t statevector_work(long long dim) { return (size_t)(4 * dim + kDenseCluster) * sizeof(double2); }

cudaError_t launch_statevector(const Engine& e, int circuit, double2* out_dev, long long dim, const int32_t* ys_dev,
                               long long nys, void* work, cudaStream_t st) {
  Engine one = e;
  one.csize = kDenseCluster;
  one.batch = 1;
  one.tc_smem = 0;
  return launch_cluster(k_dense, one, st, one, circuit, (int)dim, ys_dev, (int)nys, reinterpret_cast<double2*>(work),
                        out_dev);
}

}  // namespace gcx
