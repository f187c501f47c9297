// fp32 -> bf16 rounding of whole tensors: the donor-group gradient sums before they enter the projection GEMMs, and the
// inputs of the KVP_F32 interface (its outputs are widened by the kernels that produce them).
//
// One launch converts a whole list of tensors: a call of the fp32 interface has 3 to 5 of them per layer, each of a few
// hundred KB at the sizes that interface is for, where a launch costs more than the copy.  A four-layer training step of
// 2 x 128 tokens had 64 conversion launches of 1.6 us each, outputs included; it has 4 (device time of the step 124 -> 78
// us with a launch per list, 55 -> 52 with the outputs widened where they are produced).  Bound: HBM for large tensors,
// launch latency for small.
#include <algorithm>

#include "kvp_host.h"
#include "kvp_sm100.cuh"

namespace kvp {
namespace {

constexpr int MAX_CAST = 64;             // tensors per launch
constexpr int CAST_THREADS = 256;
constexpr int CAST_UNROLL = 4;           // 4-element pieces in flight per thread
constexpr uint32_t CAST_CHUNK = CAST_THREADS * CAST_UNROLL;   // pieces per block and turn

struct CastParams {
  const void* src[MAX_CAST];
  void* dst[MAX_CAST];
  size_t n4[MAX_CAST];                   // 4-element pieces
  uint32_t chunk_end[MAX_CAST];          // one past the tensor's last chunk in the launch's chunk order
  uint32_t chunks;
};

__global__ void __launch_bounds__(CAST_THREADS) cast_kernel(const __grid_constant__ CastParams p) {
  grid_dep_wait();
  int t = 0;
  for (uint32_t c = blockIdx.x; c < p.chunks; c += gridDim.x) {
    if (c + gridDim.x >= p.chunks) grid_dep_launch();
    while (c >= p.chunk_end[t]) ++t;
    const size_t first = size_t(c - (t ? p.chunk_end[t - 1] : 0)) * CAST_CHUNK + threadIdx.x;
    const float4* src = reinterpret_cast<const float4*>(p.src[t]);
    uint2* dst = reinterpret_cast<uint2*>(p.dst[t]);
    const size_t n4 = p.n4[t];
    float4 v[CAST_UNROLL];
#pragma unroll
    for (int u = 0; u < CAST_UNROLL; ++u)
      if (first + u * CAST_THREADS < n4) v[u] = src[first + u * CAST_THREADS];
#pragma unroll
    for (int u = 0; u < CAST_UNROLL; ++u)
      if (first + u * CAST_THREADS < n4) dst[first + u * CAST_THREADS] = make_uint2(pack_bf16(v[u].x, v[u].y), pack_bf16(v[u].z, v[u].w));
  }
}

}  // namespace

int cast_tensors(const CastItem* items, int n, cudaStream_t stream) {
  for (int i = 0; i < n; ++i)
    if ((items[i].elems & 3) != 0) return KVP_ERR_UNSUPPORTED;
  CastParams p;
  int begin = 0;
  while (begin < n) {
    uint64_t chunks = 0;
    int cnt = 0;
    for (; cnt < MAX_CAST && begin + cnt < n; ++cnt) {
      const CastItem& it = items[begin + cnt];
      const uint64_t more = (it.elems / 4 + CAST_CHUNK - 1) / CAST_CHUNK;
      if (more > 0xffffffffu) return KVP_ERR_UNSUPPORTED;
      if (chunks + more > 0xffffffffu) break;
      chunks += more;
      p.src[cnt] = it.src;
      p.dst[cnt] = it.dst;
      p.n4[cnt] = it.elems / 4;
      p.chunk_end[cnt] = uint32_t(chunks);
    }
    p.chunks = uint32_t(chunks);
    begin += cnt;
    if (chunks == 0) continue;
    const int blocks = int(std::min<uint64_t>(uint64_t(sm_count()) * 8, chunks));
    const cudaError_t e = launch_kernel(cast_kernel, blocks, CAST_THREADS, 0, stream, 1, p);
    if (e != cudaSuccess) return KVP_ERR_CUDA;
  }
  return KVP_OK;
}

}  // namespace kvp
