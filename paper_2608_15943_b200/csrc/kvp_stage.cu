// Element-wise operators of a decoder stage (RMSNorm, rotary position embedding, SwiGLU, residual add), so
// that a whole pipeline stage's forward pass can be timed with this library's kernels (the paper's stage
// tables list a forward time per stage).  All four are bound by HBM bandwidth: 16-byte accesses, fp32
// arithmetic, bf16 storage, one pass over the data, grids sized to the SM count.
#include <math.h>

#include <algorithm>

#include "kvp_host.h"
#include "kvp_rope_freq.h"
#include "kvp_sm100.cuh"

namespace kvp {
namespace {

__device__ __forceinline__ void unpack8(const uint4& v, float (&f)[8]) {
  const __nv_bfloat162* h = reinterpret_cast<const __nv_bfloat162*>(&v);
#pragma unroll
  for (int i = 0; i < 4; ++i) {
    const float2 t = __bfloat1622float2(h[i]);
    f[2 * i] = t.x;
    f[2 * i + 1] = t.y;
  }
}
__device__ __forceinline__ uint4 pack8(const float (&f)[8]) {
  return make_uint4(pack_bf16(f[0], f[1]), pack_bf16(f[2], f[3]), pack_bf16(f[4], f[5]), pack_bf16(f[6], f[7]));
}

// y = x / sqrt(mean(x^2) + eps) * w.  One CTA of 256 threads takes ROWS rows at a time, held in registers between the
// reduction and the scaling; the next rows are requested before these are reduced.  Two rows share a block barrier (one,
// since the partial sums alternate between two buffers) and the weights stay in registers: 8192 x 4096 25.3 -> 22.0 us,
// 2400 x 4096 10.2 -> 7.8.  Up to eight rows per SM go one to a CTA (347 rows 2.9 -> 2.2).  Rows of more than 4096 elements
// leave no registers for that: their weights come from L1 for every row, with four CTAs an SM up to 6144 elements and three
// up to 8192 (us, weights in registers and two CTAs -> so: 16384 x 5120 64.2 -> 52.4, 8192 x 5120 33.6 -> 27.6, 16384 x 8192
// 86.7 -> 82.5).  Bound: HBM.
constexpr int kNormThreads = 256;
constexpr int kMaxChunks = 4;  // D <= 8192
template <int CHUNKS, int ROWS>
__global__ void __launch_bounds__(kNormThreads) rmsnorm_kernel(const uint4* x, const uint4* w,
                                                               uint4* y, int T, int D8, float inv_d, float eps) {
  __shared__ float part[2][ROWS][kNormThreads / 32];
  grid_dep_wait();
  const int first = blockIdx.x * ROWS, stride = gridDim.x * ROWS;
  auto load_rows = [&](int row, uint4 (&v)[ROWS][CHUNKS]) {
#pragma unroll
    for (int r = 0; r < ROWS; ++r)
#pragma unroll
      for (int c = 0; c < CHUNKS; ++c) {
        const int i = c * kNormThreads + threadIdx.x;
        v[r][c] = make_uint4(0u, 0u, 0u, 0u);
        if (i < D8 && row + r < T) v[r][c] = x[size_t(row + r) * D8 + i];
      }
  };
  constexpr bool KEEP = CHUNKS <= 2;          // the weights in registers
  uint4 v[ROWS][CHUNKS], vn[ROWS][CHUNKS], g[CHUNKS];
  load_rows(first, v);
  auto load_weights = [&]() {
#pragma unroll
    for (int c = 0; c < CHUNKS; ++c) {
      const int i = c * kNormThreads + threadIdx.x;
      if (i < D8) g[c] = w[i];
    }
  };
  if (KEEP) load_weights();
  int buf = 0;
  for (int row = first; row < T; row += stride, buf ^= 1) {
    if (row + stride < T) load_rows(row + stride, vn);
    else grid_dep_launch();
#pragma unroll
    for (int r = 0; r < ROWS; ++r) {
      float ss = 0.f;
#pragma unroll
      for (int c = 0; c < CHUNKS; ++c) {
        float f[8];
        unpack8(v[r][c], f);
#pragma unroll
        for (int k = 0; k < 8; ++k) ss = fmaf(f[k], f[k], ss);
      }
#pragma unroll
      for (int s = 16; s > 0; s >>= 1) ss += __shfl_xor_sync(0xffffffffu, ss, s);
      if ((threadIdx.x & 31) == 0) part[buf][r][threadIdx.x >> 5] = ss;
    }
    if (!KEEP) load_weights();
    __syncthreads();
#pragma unroll
    for (int r = 0; r < ROWS; ++r) {
      float tot = 0.f;
#pragma unroll
      for (int k = 0; k < kNormThreads / 32; ++k) tot += part[buf][r][k];
      const float rs = rsqrtf(tot * inv_d + eps);
#pragma unroll
      for (int c = 0; c < CHUNKS; ++c) {
        const int i = c * kNormThreads + threadIdx.x;
        if (i < D8 && row + r < T) {
          float f[8], wt[8];
          unpack8(v[r][c], f);
          unpack8(g[c], wt);
#pragma unroll
          for (int k = 0; k < 8; ++k) f[k] = f[k] * rs * wt[k];
          y[size_t(row + r) * D8 + i] = pack8(f);
        }
      }
    }
#pragma unroll
    for (int r = 0; r < ROWS; ++r)
#pragma unroll
      for (int c = 0; c < CHUNKS; ++c) v[r][c] = vn[r][c];
  }
}

// In-place rotary embedding of x [B, S, H, dh]: pair i of every head turns by (pos0 + s) * theta^(-2i/dh).
// One thread per (token, 8 consecutive elements of the head dimension, group of heads): it forms the four rotations once
// and applies them to that slice of every head of the group, so the sines and cosines cost little beside the loads and
// stores.  The group is all heads where there are tokens enough to fill the device, fewer down to four where there are
// not: 347 tokens x 32 heads went to 22 blocks, each thread eight rounds of loads and stores one after the other (5.2 ->
// 2.3 us; 16 tokens 4.9 -> 1.7, 8192 tokens 25.3 -> 22.6).  The rotations need no memory and are formed before the kernel
// waits for the one ahead of it.
// The frequencies arrive as float pairs hi + lo (kvp_rope_freq.h); the angle pos * f is formed as an
// exact product p = pos * hi plus its rounding error and the lo term, sine and cosine of the float p are taken after an
// exact range reduction, and the small remainder is applied as a second-order correction.
constexpr int kMaxRopePairs = 128;
constexpr uint32_t kRopeUnroll = 4;
struct RopeFreq {
  float2 f[kMaxRopePairs];
};
__global__ void rope_kernel(uint4* x, uint32_t n_work, uint32_t S, uint32_t H, uint32_t dh8, uint32_t group,
                            int pos0, const __grid_constant__ RopeFreq fr) {
  // lanes of a warp need different table entries: shared memory serves them in one pass, the constant bank
  // that holds kernel parameters would replay once per distinct address
  __shared__ float2 freq[kMaxRopePairs];
  for (int k = threadIdx.x; k < int(dh8) * 4; k += blockDim.x) freq[k] = fr.f[k];
  __syncthreads();
  const uint32_t stride = gridDim.x * blockDim.x;
  const uint32_t per_tok = H * dh8, n_groups = (H + group - 1) / group;
  for (uint32_t i = blockIdx.x * blockDim.x + threadIdx.x; i < n_work; i += stride) {  // 32-bit index arithmetic only
    if (n_work - i <= stride) grid_dep_launch();
    const uint32_t c = i % dh8;                       // which group of 4 pairs inside the head
    const uint32_t h_first = i / dh8 % n_groups * group, h_end = min(H, h_first + group);
    const uint32_t tok = i / dh8 / n_groups;          // b * S + s
    const float pos = float(pos0 + int(tok % S));     // exact
    float sn2[4], cs2[4];
#pragma unroll
    for (int k = 0; k < 4; ++k) {
      const float2 fq = freq[c * 4 + k];
      const float p = pos * fq.x;
      const float d = fmaf(pos, fq.y, fmaf(pos, fq.x, -p));   // angle - p
      // p (< 2^18) reduced to [-pi, pi] with 2*pi split into three floats whose first has 8 significant
      // bits, so that k * 6.28125 is exact and the subtraction loses nothing (error about 1e-7)
      const float kk = rintf(p * 0.15915494309189535f);
      float rr = fmaf(-kk, 6.28125f, p);
      rr = fmaf(-kk, 0.00193023681640625f, rr);
      rr = fmaf(-kk, 5.070363386039389e-06f, rr);
      const float sn = __sinf(rr), cs = __cosf(rr);
      const float h = 0.5f * d * d;
      sn2[k] = sn + d * cs - h * sn;
      cs2[k] = cs - d * sn - h * cs;
    }
    uint4* const base = x + size_t(tok) * per_tok + c;
    constexpr uint32_t UNROLL = kRopeUnroll;          // loads in flight per thread
    grid_dep_wait();
    for (uint32_t h0 = h_first; h0 < h_end; h0 += UNROLL) {
      uint4 v[UNROLL];
#pragma unroll
      for (uint32_t u = 0; u < UNROLL; ++u)
        if (h0 + u < h_end) v[u] = base[size_t(h0 + u) * dh8];
#pragma unroll
      for (uint32_t u = 0; u < UNROLL; ++u) {
        if (h0 + u < h_end) {
          float f[8];
          unpack8(v[u], f);
#pragma unroll
          for (int k = 0; k < 4; ++k) {
            const float a = f[2 * k], b = f[2 * k + 1];
            f[2 * k] = a * cs2[k] - b * sn2[k];
            f[2 * k + 1] = a * sn2[k] + b * cs2[k];
          }
          base[size_t(h0 + u) * dh8] = pack8(f);
        }
      }
    }
  }
}

// out = silu(gate) * up
// out[i] = f(a[i], b[i]) over 16-byte pieces.  TWO: a thread has at most two, with all four loads in flight.  Up to that
// size the bound is the latency of the loads, beyond it memory.  Measured (us, a loop -> TWO): add 16 x 4096 1.23 -> 1.15,
// 347 x 4096 2.57 -> 1.65, 652 x 5504 3.91 -> 3.22; swiglu 347 x 11008 5.44 -> 5.24, but 16 x 4096 1.74 -> 1.81 (more
// set-up), so that it takes the loop where a thread has a single piece.  Both stay within 32 registers: with 48, five
// blocks an SM instead of eight, swiglu of 8192 x 4096 took 37.2 instead of 33.4.
template <bool TWO, typename F>
__device__ __forceinline__ void zip8(const uint4* a, const uint4* b, uint4* out, size_t n8, F f) {
  const size_t stride = size_t(gridDim.x) * blockDim.x;
  size_t i = size_t(blockIdx.x) * blockDim.x + threadIdx.x;
  auto piece = [&](const uint4& p, const uint4& q) {
    float x[8], y[8];
    unpack8(p, x);
    unpack8(q, y);
#pragma unroll
    for (int k = 0; k < 8; ++k) x[k] = f(x[k], y[k]);
    return pack8(x);
  };
  if constexpr (TWO) {
    if (i >= n8) return;
    const uint4 a0 = a[i], b0 = b[i];
    const bool more = i + stride < n8;
    uint4 a1 = a0, b1 = b0;
    if (more) {
      a1 = a[i + stride];
      b1 = b[i + stride];
    }
    grid_dep_launch();
    out[i] = piece(a0, b0);
    if (more) out[i + stride] = piece(a1, b1);
  } else {
    for (; i < n8; i += stride) {
      if (i + stride >= n8) grid_dep_launch();
      const uint4 a0 = a[i], b0 = b[i];
      out[i] = piece(a0, b0);
    }
  }
}

constexpr int kStreamThreads = 256, kStreamResident = 8;   // CTAs per SM
// The correctly rounded reciprocal at every size: an element's result depends on its two inputs alone.  (rcp.approx, up to an ulp
// off, is a dozen instructions less, but moves results that lie near a tie of the bf16 rounding, five in a million.  It gained
// 0.5 to 1.0 us a launch up to sixteen pieces a thread, 16 x 11008 1.73 -> 1.27, 2048 x 11008 22.6 -> 21.7, and lost beyond.)
template <bool TWO>
__global__ void __launch_bounds__(kStreamThreads, kStreamResident)
    swiglu_kernel(const uint4* gate, const uint4* up, uint4* out, size_t n8) {
  grid_dep_wait();
  zip8<TWO>(gate, up, out, n8, [](float g, float u) { return g * __frcp_rn(1.f + __expf(-g)) * u; });
}

template <bool TWO>
__global__ void __launch_bounds__(kStreamThreads, kStreamResident)
    add_kernel(const uint4* a, const uint4* b, uint4* out, size_t n8) {
  grid_dep_wait();
  zip8<TWO>(a, b, out, n8, [](float x, float y) { return x + y; });
}

bool is_aligned16(const void* p) { return (reinterpret_cast<uintptr_t>(p) & 15) == 0; }
int streaming_blocks(size_t n8) { return int(min(size_t(sm_count()) * kStreamResident, (n8 + kStreamThreads - 1) / kStreamThreads)); }
size_t one_round() { return size_t(sm_count()) * kStreamResident * kStreamThreads; }   // pieces

}  // namespace
}  // namespace kvp

using namespace kvp;

extern "C" int kvp_rmsnorm(int32_t T, int32_t D, const void* x, const void* w, float eps, void* y, kvp_stream_t stream) {
  if (T < 0 || D < 1 || x == nullptr || w == nullptr || y == nullptr || !(eps >= 0.f)) return KVP_ERR_INVALID_ARG;
  if (D % 8 != 0 || D > 8 * kNormThreads * kMaxChunks || !is_aligned16(x) || !is_aligned16(w) || !is_aligned16(y)) return KVP_ERR_UNSUPPORTED;
  if (T == 0) return KVP_OK;
  const int d8 = D / 8, sms = sm_count();
  const int chunks = (d8 + kNormThreads - 1) / kNormThreads;
  const bool two = T > 8 * sms && chunks <= 2;   // wider rows: the registers of two would leave one CTA per SM
  auto* const kernel = chunks == 1 ? (two ? rmsnorm_kernel<1, 2> : rmsnorm_kernel<1, 1>)
                       : chunks == 2 ? (two ? rmsnorm_kernel<2, 2> : rmsnorm_kernel<2, 1>)
                       : chunks == 3 ? rmsnorm_kernel<3, 1>
                                     : rmsnorm_kernel<kMaxChunks, 1>;
  const int resident = chunks == 1 ? 5 : chunks == 2 ? 3 : chunks == 3 ? 4 : 3;   // CTAs per SM by registers
  const int blocks = T <= 8 * sms && chunks <= 2 ? T : std::min(two ? (T + 1) / 2 : T, sms * resident);
  const cudaError_t e = launch_kernel(kernel, blocks, kNormThreads, 0, reinterpret_cast<cudaStream_t>(stream), 1,
      reinterpret_cast<const uint4*>(x), reinterpret_cast<const uint4*>(w), reinterpret_cast<uint4*>(y), T, d8, 1.f / float(D), eps);
  return e == cudaSuccess ? KVP_OK : KVP_ERR_CUDA;
}

extern "C" int kvp_rope(int32_t B, int32_t S, int32_t H, int32_t dh, float theta, int32_t pos0, void* x, kvp_stream_t stream) {
  if (B < 0 || S < 0 || H < 1 || dh < 2 || x == nullptr || !(theta > 1.f) || pos0 < 0) return KVP_ERR_INVALID_ARG;
  if (dh % 8 != 0 || dh / 2 > kMaxRopePairs || !is_aligned16(x) || int64_t(pos0) + S > (int64_t(1) << 18)) return KVP_ERR_UNSUPPORTED;
  const size_t n8 = size_t(B) * S * H * (dh / 8);
  if (n8 == 0) return KVP_OK;
  RopeFreq fr;
  static_assert(sizeof(float2) == 2 * sizeof(float), "hi and lo of a pair lie side by side");
  rope_frequencies(double(theta), dh, &fr.f[0].x, &fr.f[0].y, 2);
  // 16-byte groups are indexed with 32 bits: larger tensors go in slices of whole sequences
  const size_t per_seq = size_t(S) * H * (dh / 8);
  if (per_seq >= (size_t(1) << 31)) return KVP_ERR_UNSUPPORTED;
  const int seqs_per_launch = int(std::max<size_t>(1, ((size_t(1) << 31) - 1) / per_seq));
  for (int b0 = 0; b0 < B; b0 += seqs_per_launch) {
    const size_t slices = size_t(std::min(seqs_per_launch, B - b0)) * S * (dh / 8);   // (token, 8-element slice)
    uint32_t group = uint32_t(H);
    while (group > kRopeUnroll && slices * ((H + group - 1) / group) < size_t(sm_count()) * 1024) group = (group + 1) / 2;
    const uint32_t n_work = uint32_t(slices * ((H + group - 1) / group));
    const cudaError_t e = launch_kernel(rope_kernel, streaming_blocks(n_work), kStreamThreads, 0, reinterpret_cast<cudaStream_t>(stream), 1,
        reinterpret_cast<uint4*>(x) + size_t(b0) * per_seq, n_work, uint32_t(S), uint32_t(H), uint32_t(dh / 8), group, pos0, fr);
    if (e != cudaSuccess) return KVP_ERR_CUDA;
  }
  return KVP_OK;
}

extern "C" int kvp_swiglu(int64_t n, const void* gate, const void* up, void* out, kvp_stream_t stream) {
  if (n < 0 || gate == nullptr || up == nullptr || out == nullptr) return KVP_ERR_INVALID_ARG;
  if (n % 8 != 0 || !is_aligned16(gate) || !is_aligned16(up) || !is_aligned16(out)) return KVP_ERR_UNSUPPORTED;
  if (n == 0) return KVP_OK;
  const size_t n8 = size_t(n / 8);
  const cudaError_t e = launch_kernel(n8 > one_round() && n8 <= 2 * one_round() ? swiglu_kernel<true> : swiglu_kernel<false>, streaming_blocks(n8),
      kStreamThreads, 0, reinterpret_cast<cudaStream_t>(stream), 1,
      reinterpret_cast<const uint4*>(gate), reinterpret_cast<const uint4*>(up), reinterpret_cast<uint4*>(out), n8);
  return e == cudaSuccess ? KVP_OK : KVP_ERR_CUDA;
}

extern "C" int kvp_add(int64_t n, const void* a, const void* b, void* out, kvp_stream_t stream) {
  if (n < 0 || a == nullptr || b == nullptr || out == nullptr) return KVP_ERR_INVALID_ARG;
  if (n % 8 != 0 || !is_aligned16(a) || !is_aligned16(b) || !is_aligned16(out)) return KVP_ERR_UNSUPPORTED;
  if (n == 0) return KVP_OK;
  const cudaError_t e = launch_kernel(size_t(n / 8) <= 2 * one_round() ? add_kernel<true> : add_kernel<false>, streaming_blocks(size_t(n / 8)), kStreamThreads, 0, reinterpret_cast<cudaStream_t>(stream), 1,
      reinterpret_cast<const uint4*>(a), reinterpret_cast<const uint4*>(b), reinterpret_cast<uint4*>(out), size_t(n / 8));
  return e == cudaSuccess ? KVP_OK : KVP_ERR_CUDA;
}
