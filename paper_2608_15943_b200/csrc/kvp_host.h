// Host-side helpers shared by the translation units of the library (not part of the C ABI).
#pragma once
#include <cuda.h>
#include <cuda_runtime.h>
#include <stddef.h>
#include <stdint.h>

#include <atomic>

#include "../../include/kvp.h"

namespace kvp {

// Builds a tiled TMA descriptor over a row-major bf16/fp32 tensor of up to 4 dimensions.
// dims[0] is the innermost (contiguous) extent in elements; strides_bytes[i] is the byte stride
// of dims[i+1].  box[] is the tile copied per request.  swizzle128 selects the 128-byte swizzle
// (the inner box extent must then span exactly 128 bytes).  Returns KVP_OK or KVP_ERR_CUDA.
int make_tensor_map(CUtensorMap* out, const void* base, int elem_bytes, int rank, const uint64_t* dims,
                    const uint64_t* strides_bytes, const uint32_t* box, bool swizzle128);

inline bool aligned16(const void* p) { return (reinterpret_cast<uintptr_t>(p) & 15u) == 0; }

// Types of C: bf16; the fp32 sums; the sums rounded to bf16 and stored as fp32 (the fp32 interface's outputs).
enum { OUT_BF16 = 0, OUT_F32 = 1, OUT_F32_OF_BF16 = 2 };

// One GEMM "segment": C += op(A) * op(B) over this segment's K extent.
struct GemmSeg {
  const void* a;   // bf16
  const void* b;   // bf16
  int64_t lda;     // elements: row stride of the stored matrix
  int64_t ldb;
  int K;
};

// C[M,N] = sum over segments of A_s * B_s, bf16 inputs, fp32 accumulation in TMEM.
//   a_mn == 0: A_s stored [M, K] row-major (K-major);  a_mn == 1: stored [K, M] row-major.
//   b_mn == 0: B_s stored [N, K] row-major (K-major);  b_mn == 1: stored [K, N] row-major.
//   out_f32: type of C (OUT_*); ldc in elements.
// withhold_at / wait_limit_ns serve the self-test of the bounded waits (kvp_selftest_bounded_wait) only.
int gemm_bf16(int M, int N, const GemmSeg* segs, int nseg, int a_mn, int b_mn, void* c, int64_t ldc, int out_f32,
              cudaStream_t stream, int withhold_at = 0, unsigned long long wait_limit_ns = 0);

// One problem of a grouped launch: C[M,N] = sum over segments, with its own operand modes and output type.
struct GemmProblem {
  int M, N;
  GemmSeg segs[3];
  int nseg;
  int a_mn, b_mn;
  void* c;
  int64_t ldc;
  int out_f32;
};

// All problems in as few launches as the kernel's parameter block allows (32 problems and 48 segments per launch);
// the tiles are walked in the order of the list, so the problems with the longest tiles should come first.
// Which kernel a launch takes follows from its sizes and operand modes (kvp_gemm.cu).
int gemm_grouped(const GemmProblem* probs, int n, cudaStream_t stream);

// fp32 -> bf16 (round-to-nearest-even) of a list of tensors in as few launches as the parameter block allows.  elems:
// multiples of 4.
struct CastItem {
  const void* src;   // fp32
  void* dst;         // bf16
  size_t elems;
};
int cast_tensors(const CastItem* items, int n, cudaStream_t stream);

// The attention backward of the fp32 interface: dO as the caller has it (O is in either interface), and what else is to be rounded.
struct BwdF32 {
  const float* const* d_o;
  const CastItem* casts;
  int n_casts;
  bool read_first;   // all inputs are read before any output is written
};

void gemm_set_pair_mode(int mode);   // 0: single-CTA tiles only, 1: pairs where the caller prefers them, 2: pairs everywhere
int gemm_pair_mode();
int gemm_read_status();
int attn_fwd_read_status();
int attn_bwd_read_status();
int decode_read_status();

int sm_count();

// Bookkeeping for benchmarks: every kernel launch of the library is counted, and a caller may
// ask for CUDA events to be recorded around the launches of one named kernel.
enum {
  KVP_KERNEL_GEMM = 0,
  KVP_KERNEL_ATTN_FWD = 1,
  KVP_KERNEL_ATTN_BWD = 2,      // single-pass backward kernel (dQ partials, dK, dV)
  KVP_KERNEL_DECODE = 3,
  KVP_KERNEL_ATTN_BWD_AUX = 4,  // backward helper passes: Delta, accumulator clear, dQ conversion
  KVP_KERNEL_COUNT = 5
};
void note_launch(int n = 1);

// Raises a kernel's dynamic shared-memory limit, once per device.
template <auto Kernel>
cudaError_t allow_smem(int bytes) {
  static std::atomic<uint64_t> done{0};
  int dev = 0;
  cudaError_t e = cudaGetDevice(&dev);
  if (e != cudaSuccess) return e;
  const uint64_t bit = uint64_t(1) << (dev & 63);
  if (dev < 64 && (done.load(std::memory_order_relaxed) & bit) != 0) return cudaSuccess;
  e = cudaFuncSetAttribute(Kernel, cudaFuncAttributeMaxDynamicSharedMemorySize, bytes);
  if (e == cudaSuccess && dev < 64) done.fetch_or(bit, std::memory_order_relaxed);
  return e;
}

template <typename T>
struct SameType { using type = T; };   // keeps the argument types of launch_kernel out of template deduction

// Every kernel of the library is launched through this: programmatic stream serialisation lets its CTAs come up (barriers,
// tensor-memory allocation, descriptor fetches) while the kernel before it on the stream drains.  The kernel must
// execute grid_dep_wait() before it relies on or changes global memory (decode and its merge look at the lengths ahead of it,
// and again behind it), and grid_dep_launch() so that the next kernel may do the same:
// the long ones when their last loads are out, the short ones (split GEMM, cache append, merge of decode pieces) as soon as
// a CTA is set up.  (Any thread's grid_dep_launch() counts for its CTA.  Given at set-up by the long ones too, it parked
// the next kernel's CTAs on the SMs for the whole of each, and the 46 ms training step of 2 x 8192 tokens took 1.2 ms
// longer.)  cluster > 1 sets a runtime cluster size.  Device time of a pass (graph replay), plain
// launches -> these: tiny fp32 training step 59.4 -> 54.4 us, token step of a four-layer stage 635 -> 588 us (56
// kernels), prompt of 347 tokens through it 1064 -> 1031 us.
template <typename... KP>
cudaError_t launch_kernel(void (*kernel)(KP...), dim3 grid, dim3 block, size_t smem, cudaStream_t stream, int cluster,
                          const typename SameType<KP>::type&... args) {
  cudaLaunchAttribute at[2];
  at[0].id = cudaLaunchAttributeProgrammaticStreamSerialization;
  at[0].val.programmaticStreamSerializationAllowed = 1;
  at[1].id = cudaLaunchAttributeClusterDimension;
  at[1].val.clusterDim.x = unsigned(cluster);
  at[1].val.clusterDim.y = at[1].val.clusterDim.z = 1;
  cudaLaunchConfig_t lc = {};
  lc.gridDim = grid;
  lc.blockDim = block;
  lc.dynamicSmemBytes = smem;
  lc.stream = stream;
  lc.attrs = at;
  lc.numAttrs = cluster > 1 ? 2 : 1;
  void* ptrs[] = {const_cast<void*>(static_cast<const void*>(&args))...};
  note_launch();
  return cudaLaunchKernelExC(&lc, reinterpret_cast<const void*>(kernel), ptrs);
}

void timing_before(int kernel, cudaStream_t stream);
void timing_after(int kernel, cudaStream_t stream);

}  // namespace kvp
