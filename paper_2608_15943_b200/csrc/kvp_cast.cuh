// fp32 -> bf16 rounding of a list of tensors: what a launch of kvp_misc.cu does, and the backward's pre-pass of the fp32
// interface beside its own work.
#pragma once

#include <algorithm>

#include "kvp_host.h"
#include "kvp_sm100.cuh"

namespace kvp {

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

// The blocks of the launch that convert: `blocks` of them, this one the block-th, of CAST_THREADS threads.
__device__ __forceinline__ void cast_chunks(const CastParams& p, uint32_t block, uint32_t blocks) {
  int t = 0;
  for (uint32_t c = block; c < p.chunks; c += blocks) {
    if (c + blocks >= p.chunks) grid_dep_launch();
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

// Takes items from the front of the list until the parameter block is full; how many.
inline int fill_casts(CastParams& p, const CastItem* items, int n) {
  uint64_t chunks = 0;
  int cnt = 0;
  for (; cnt < MAX_CAST && cnt < n; ++cnt) {
    const CastItem& it = items[cnt];
    const uint64_t more = (it.elems / 4 + CAST_CHUNK - 1) / CAST_CHUNK;
    if (more > 0xffffffffu || chunks + more > 0xffffffffu) break;
    chunks += more;
    p.src[cnt] = it.src;
    p.dst[cnt] = it.dst;
    p.n4[cnt] = it.elems / 4;
    p.chunk_end[cnt] = uint32_t(chunks);
  }
  p.chunks = uint32_t(chunks);
  return cnt;
}

}  // namespace kvp
