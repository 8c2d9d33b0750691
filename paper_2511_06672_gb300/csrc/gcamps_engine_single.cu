// Single-operation launches of libgcamps (arxiv 2511.06672, Sec. 3): one Clifford gate, one non-Clifford
// step or one disentangling sweep on every circuit of a handle.

#include "gcamps_device.cuh"

namespace gcx {
namespace {

__global__ void __launch_bounds__(kThreads, kMinCtas) k_single(Engine e, gcamps_op op) { single_body(e, op); }

// One Clifford gate on every circuit: only the tableaux, so a CTA a circuit and no cluster.
__global__ void __launch_bounds__(kThreads) k_clifford(Engine e, gcamps_op op) {
  __shared__ Smem s;
  const long long t0 = clock64();
  Ctx C = make_ctx(e, blockIdx.x);
  apply_cliffords(s, C, &op, 1);
  if (threadIdx.x == 0) {
    C.stats[S_CLIFF] += 1;
    C.prof[P_CLIFF] += clock64() - t0;
  }
}

}  // namespace

cudaError_t launch_single(const Engine& e, const gcamps_op& op, cudaStream_t st) {
  if (op.kind == GCAMPS_OP_CLIFFORD) {
    k_clifford<<<e.batch, kThreads, 0, st>>>(e, op);
    return cudaGetLastError();
  }
  if (e.precision) return launch_single_tc(e, op, st);
  return launch_cluster(k_single, e, st, e, op);
}

}  // namespace gcx
