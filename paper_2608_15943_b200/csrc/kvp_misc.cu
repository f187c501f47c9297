// fp32 -> bf16 rounding of whole tensors: the donor-group gradient sums before they enter the projection GEMMs, and the
// inputs of the KVP_F32 interface (its outputs are widened by the kernels that produce them).
//
// One launch converts a whole list of tensors: a call of the fp32 interface has 3 to 5 of them per layer, each of a few
// hundred KB at the sizes that interface is for, where a launch costs more than the copy.  A four-layer training step of
// 2 x 128 tokens had 64 conversion launches of 1.6 us each, outputs included; it has 3, and the backward's pre-pass converts
// beside its own work (kvp_cast.cuh; device time of the step 124 -> 78
// us with a launch per list, 55 -> 52 with the outputs widened where they are produced).  Bound: HBM for large tensors,
// launch latency for small.
#include <algorithm>

#include "kvp_cast.cuh"

namespace kvp {
namespace {

__global__ void __launch_bounds__(CAST_THREADS) cast_kernel(const __grid_constant__ CastParams p) {
  grid_dep_wait();
  cast_chunks(p, blockIdx.x, gridDim.x);
}

}  // namespace

int cast_tensors(const CastItem* items, int n, cudaStream_t stream) {
  for (int i = 0; i < n; ++i)
    if ((items[i].elems & 3) != 0) return KVP_ERR_UNSUPPORTED;
  CastParams p;
  int begin = 0;
  while (begin < n) {
    const int cnt = fill_casts(p, items + begin, n - begin);
    if (cnt == 0) return KVP_ERR_UNSUPPORTED;   // a tensor of more chunks than the list can count
    begin += cnt;
    if (p.chunks == 0) continue;
    const int blocks = int(std::min<uint64_t>(uint64_t(sm_count()) * 8, p.chunks));
    const cudaError_t e = launch_kernel(cast_kernel, blocks, CAST_THREADS, 0, stream, 1, p);
    if (e != cudaSuccess) return KVP_ERR_CUDA;
  }
  return KVP_OK;
}

}  // namespace kvp
