// Flash-attention backward over a donor map (chain rule of Eq. 2-3 of the paper) in ONE pass.
//
//  bwd_kernel   KV-stationary.  One CTA owns a 128-row K/V tile of one (batch, KV head) of a DONOR
//               layer, keeps K and V in shared memory and the dK / dV accumulators in TMEM (fp32)
//               while it walks the query streams that read the tile: the donor itself and all its
//               consumer layers, the Hq/Hkv query heads of the KV head's group, and a window of the 64-row
//               query tiles the causal mask lets see the keys.  dK and dV of the donor are therefore summed
//               on chip across layers and heads and added to the fp32 sums in HBM once per CTA; where a key
//               tile has several (windows, and parts of the streams in small calls), in no fixed order.  Per step, transposed so that TMEM
//               lane == key row:  S^T = K Q^T, dP^T = V dO^T (tcgen05; K and V from TMEM at DH 64), each
//               followed by one rank-3 MMA that subtracts the query's LSE/scale resp. Delta (a bf16
//               three-term split against a tile of ones), so the accumulators already hold the
//               exponent and dP - Delta; P^T = exp2(c acc), dS^T = P^T acc' are written back as bf16
//               over the score columns and fed to dV += P^T dO, dK += dS^T Q as the A operand FROM
//               TMEM.  dS^T also goes to shared memory, where it is the B operand of the fifth product
//               dQ^T = K^T dS^T (K read as an MN-major A operand): the step's [dh x 64] partial of dQ
//               lands in TMEM, a third warpgroup moves it to shared memory and adds it to an fp32
//               accumulator in global memory with bulk reductions (cp.reduce.async.bulk .add.f32, 8 KB
//               each), so S and dP are computed once for all three gradients.
//
//  dq_convert_kernel  scales the fp32 dQ accumulators and writes dQ as bf16 [B,S,Hq,dh].  (Up to 128 tokens a dQ tile has one
//               partial, which bwd_kernel writes as dQ itself, unless dQ lies over inputs that other CTAs may still read.)
//
// Delta = rowsum(dO * O) comes from a small pre-pass.  The dQ accumulators live in the caller's
// workspace in a blocked layout ([b][hq][64-query tile][32-column quarter][16][32 columns][4 queries] fp32) so that every
// reduction is one contiguous 8 KB run; they, and the dK / dV sums, are cleared by the pre-pass of each launch.  The
// order in which partials reach an accumulator is not fixed, so dQ, dK and dV are reproducible only up to fp32 rounding
// order (bit for bit up to 128 tokens, where no element has more than two terms).
#include <math.h>

#include <algorithm>
#include <vector>

#include "kvp_bwd_shape.h"
#include "kvp_cast.cuh"

namespace kvp {
namespace {

constexpr int BT = BWD_KEYS;        // key rows per tile
constexpr int BQ2 = BWD_QUERIES;    // query rows per step
constexpr int MAX_CLASSES = 128;
constexpr int MAX_GROUP = 8;  // layers of one donor group per launch
constexpr uint32_t HALF_BYTES = 128 * 128;  // [128 rows x 128 B] block
constexpr uint32_t QHALF_BYTES = 64 * 128;  // [ 64 rows x 128 B] block

__device__ int g_bwd_status;

__device__ __forceinline__ float fast_exp2(float x) {
  float y;
  asm("ex2.approx.ftz.f32 %0, %1;" : "=f"(y) : "f"(x));
  return y;
}

// warp 0 TMA, warp 1 MMA, warps 2-5 and 6-9 two compute warpgroups, warps 10-13 dQ drain, warps 14 and 15 statistics
// Bound at DH 128: the shared-memory port (1760 of about 1900 cycles a step).  At DH 64 a step has half the MMA work and the
// same exponentials, and the serial part of a compute warpgroup's step counts: there the warpgroups take every other step,
// which their own buffers of dP^T, dS^T and staged dQ allow.  Measured (us, whole attn_bwd call, as DH 128 -> so): 2 layers of 4 x
// 2048, 16 heads on 8, 325 -> 275; 8192, 32 heads on 8, 1020 -> 860; three layers of 3 x 776, 16 heads on 4, 89 -> 75.
constexpr int BWD_THREADS = 512;
constexpr int STAT_BYTES = 2 * BQ2 * 16;      // the statistics of 64 queries: [lse, delta][64][8] bf16
constexpr int DQ_STAGE_BYTES = BQ2 * 32 * 4;  // one drain warp's share of a step: [64 queries x 32 columns] fp32
template <int DH>
struct BwdSmem {
  static constexpr bool SMALL = DH == 64;   // TMEM and shared memory have room for more
  static constexpr int STAGES = SMALL ? 5 : 3;            // ring of (Q, dO) 64-row tiles
  static constexpr int DS_BUFS = SMALL ? 2 : 1;
  static constexpr int STEP_THREADS = SMALL ? 128 : 256;  // compute threads that work on a step
  static constexpr int DQ_BUFS = SMALL ? 2 : 1;           // staging buffers of a drain warp (two of the four have work at DH 64)
  static constexpr int KV_TILE = BT * DH * 2;
  static constexpr int Q_TILE = BQ2 * DH * 2;
  static constexpr int STAGE = 2 * Q_TILE;  // Q then dO
  static constexpr int OFF_K = 0;
  static constexpr int OFF_V = OFF_K + KV_TILE;
  static constexpr int OFF_RING = OFF_V + KV_TILE;
  static constexpr int OFF_DS = OFF_RING + STAGES * STAGE;         // dS^T [128 keys x 64 queries] bf16, 128-B swizzle
  static constexpr int OFF_DQ = OFF_DS + DS_BUFS * BT * BQ2 * 2;   // [4 drain warps][64 x 32] fp32
  static constexpr int OFF_ONES = OFF_DQ + 4 * DQ_STAGE_BYTES;     // [128 x 8] bf16: columns 0-7 of the tile of ones
  static constexpr int OFF_STAT = OFF_ONES + 2048;                 // [STAGES][lse, delta][64 x 8] bf16: columns 0-7
  static constexpr int OFF_ZERO = OFF_STAT + STAGES * STAT_BYTES;  // [128 x 8] zeros: columns 8-15 of all of the above
  static constexpr int OFF_BAR = OFF_ZERO + 2048;
  static constexpr int TOTAL = OFF_BAR + 256 + 1024;
};

// One launch serves several donor groups (up to MAX_GROUP member layers in all): slot i of the per-layer arrays is
// the i-th member layer, group g owns slots [first_slot[g], first_slot[g + 1]) and blocks [cta_begin[g],
// cta_begin[g + 1]).  Groups are sorted by size, largest first, so that only the last, shortest CTAs of the whole
// backward pass run on a partly idle device.
struct BwdParams {
  CUtensorMap map_k[MAX_GROUP], map_v[MAX_GROUP];   // per group: donor K, V [B,S,Hkv,dh], box rows 128
  CUtensorMap map_q[MAX_GROUP], map_do[MAX_GROUP];  // per member layer, box rows 64
  const float* lse[MAX_GROUP];    // [B,Hq,S]
  const float* delta[MAX_GROUP];  // [B,Hq,S]
  float* dq_acc[MAX_GROUP];       // blocked fp32 accumulators, see dq_acc_floats()
  void* dq[MAX_GROUP];            // dQ itself, [B,S,Hq,dh], bf16 or (dq_f32) the bf16 values as fp32
  int dq_f32;
  int dq_direct;                  // a dQ tile has one partial, and this kernel writes it (one key tile)
  CUtensorMap map_dk[MAX_GROUP], map_dv[MAX_GROUP]; // per group: the fp32 sums [B,S,Hkv,dh], box 32 rows x 32 columns
  int first_slot[MAX_GROUP + 1];
  int cta_begin[MAX_GROUP + 1];
  int window[MAX_GROUP];          // query tiles per CTA
  int parts[MAX_GROUP];           // parts the query streams of a (window, key tile) are dealt out in
  int ctas_per_pair[MAX_GROUP];   // CTAs of one (batch, KV head): parts x sum over windows of the key tiles that see the window
  // Longest CTAs first (small launches): classes of CTAs with the same (group, window, key tile), hence the same number of
  // steps; class c holds blocks [class_end[c - 1], class_end[c]), (batch, KV head) and part inside.  0: in index order.
  int n_classes;
  uint16_t class_end[MAX_CLASSES];
  uint32_t class_id[MAX_CLASSES];   // group << 24 | window << 12 | key tile
  int n_groups;
  int B, S, Hq, Hkv;
  int causal;
  float scale;
  float scale_log2;
};

// Unswizzled K-major operand tile of 16 bf16 per row: two halves of 8 columns, each half stored as
// rows of 16 bytes (8 rows = one 128-byte core matrix).  SBO = 128, LBO = rows * 16.
__host__ __device__ constexpr uint32_t desc_hi_plain(uint32_t sbo_bytes) { return ((sbo_bytes >> 4) & 0x3FFF) | (1u << 14); }
__device__ __forceinline__ uint32_t desc_lo_plain(uint32_t saddr, uint32_t lbo_bytes) {
  return ((saddr & 0x3FFFF) >> 4) | (((lbo_bytes >> 4) & 0x3FFF) << 16);
}
// v = h + m + l with h, m, l bf16: 24 significant bits, so a bf16 MMA can add v exactly enough
__device__ __forceinline__ uint4 split3_bf16(float v) {
  const __nv_bfloat16 h = __float2bfloat16_rn(v);
  const float r1 = v - __bfloat162float(h);
  const __nv_bfloat16 m = __float2bfloat16_rn(r1);
  const __nv_bfloat16 l = __float2bfloat16_rn(r1 - __bfloat162float(m));
  uint4 out;
  out.x = uint32_t(__bfloat16_as_ushort(h)) | (uint32_t(__bfloat16_as_ushort(m)) << 16);
  out.y = uint32_t(__bfloat16_as_ushort(l));
  out.z = 0u;
  out.w = 0u;
  return out;
}

// Eight columns from element `at` of dQ on: bf16, or the bf16 values as fp32.
__device__ __forceinline__ void store_dq(void* dq, int f32, size_t at, const uint4& v) {
  if (f32) {
    float* out = reinterpret_cast<float*>(dq) + at;
    *reinterpret_cast<uint4*>(out) = make_uint4(v.x << 16, v.x & 0xffff0000u, v.y << 16, v.y & 0xffff0000u);
    *reinterpret_cast<uint4*>(out + 4) = make_uint4(v.z << 16, v.z & 0xffff0000u, v.w << 16, v.w & 0xffff0000u);
  } else {
    *reinterpret_cast<uint4*>(reinterpret_cast<__nv_bfloat16*>(dq) + at) = v;
  }
}

// Floats of one layer's dQ accumulator: [B][Hq][ceil(S/64)][DH/32][16][32][4].
__host__ __device__ inline size_t dq_acc_floats(int B, int S, int Hq, int dh) {
  return size_t(B) * Hq * ((S + BQ2 - 1) / BQ2) * BQ2 * dh;
}

// TMEM columns: S^T of step parity i at [i*64, i*64+64) (P^T and dS^T overwrite it as bf16), then dP^T, the step's dQ^T (64),
// dK and dV (DH each).  At DH 64 dP^T too has a buffer for each parity, and K and V follow as bf16 A operands of S^T and dP^T:
// an MMA whose A comes from TMEM reads 2 KB of shared memory instead of 6, 32 cycles instead of 48.
//
// The per-query statistics are applied BY THE TENSOR CORE: one extra K-step multiplies a [128 x 16] tile
// of ones (first three columns) with a [64 x 16] tile holding -LSE/scale (resp. -Delta) of each query
// split into three bf16 terms, so the accumulators already hold S - LSE/scale and dP - Delta and the
// threads need no per-column operand: P^T = exp2(c * acc), dS^T = P^T * acc'.
template <int DH>
__global__ void __launch_bounds__(BWD_THREADS, 1) bwd_kernel(const __grid_constant__ BwdParams p) {
  using L = BwdSmem<DH>;
  constexpr int HALVES = DH / 64;
  constexpr int KSTEPS_DH = DH / 16;
  constexpr int KSTEPS_Q = BQ2 / 16;
  constexpr int KSTEPS_KV = BT / 16;

  extern __shared__ uint8_t smem_raw[];
  uint8_t* smem = reinterpret_cast<uint8_t*>((reinterpret_cast<uintptr_t>(smem_raw) + 1023) & ~uintptr_t(1023));
  uint64_t* bars = reinterpret_cast<uint64_t*>(smem + L::OFF_BAR);
  uint64_t* kv_full = bars + 0;
  uint64_t* q_full = bars + 1;                    // [STAGES] Q and dO loaded, statistics staged (64 arrivals)
  uint64_t* q_empty = q_full + L::STAGES;         // [STAGES]
  uint64_t* st_full = q_empty + L::STAGES;        // [2] S^T and dP^T of the step are in TMEM
  uint64_t* dp_free = st_full + 2;                // [2] dP^T of the step is in registers (STEP_THREADS arrivals)
  uint64_t* pds_ready = dp_free + 2;              // [2] P^T, dS^T written (TMEM and shared memory; STEP_THREADS arrivals)
  uint64_t* dq_full = pds_ready + 2;              // [2] dQ^T of the step is in TMEM; its dS^T tile may be overwritten
  uint64_t* dq_free = dq_full + 2;                // dQ^T of the step is in registers (128 arrivals)
  uint64_t* acc_done = dq_free + 1;               // all MMAs have completed
  uint64_t* a_ready = acc_done + 1;               // DH 64: K and V are in TMEM (256 arrivals)
  uint32_t* tmem_slot = reinterpret_cast<uint32_t*>(a_ready + 1);

  const int warp = threadIdx.x >> 5;
  const int lane = threadIdx.x & 31;
  int* err = &g_bwd_status;

  // Work decomposition.  A CTA is one donor group, one (batch, KV head), one 128-row key tile and one WINDOW of
  // consecutive 64-row query tiles, for every query stream of the donor group.  All CTAs therefore take
  // (nearly) the same number of steps per stream and walk the streams at the same pace, so the CTAs that
  // run at the same time read the same few Q / dO tiles and add to the same few dQ accumulator tiles:
  // what a wave touches over its lifetime stays in L2.  Blocks are dispatched in index order: (batch, KV
  // head) slowest, then the window, then the key tiles that see it.  The windows of one key tile add their
  // dK / dV partials to the (cleared) output with reductions.
  const int n_jt = (p.S + BT - 1) / BT;
  const int n_qt = (p.S + BQ2 - 1) / BQ2;
  int grp = 0, jt = 0, win = 0, pair = 0, part = 0;
  if (p.n_classes > 0) {
    int lo = 0, hi = p.n_classes - 1;
    while (lo < hi) {
      const int mid = (lo + hi) / 2;
      if (int(blockIdx.x) < p.class_end[mid]) hi = mid;
      else lo = mid + 1;
    }
    const uint32_t id = p.class_id[lo];
    grp = id >> 24;
    win = (id >> 12) & 0xfff;
    jt = id & 0xfff;
    const int in_class = int(blockIdx.x) - (lo ? p.class_end[lo - 1] : 0);
    pair = in_class / p.parts[grp];
    part = in_class - pair * p.parts[grp];
  } else {
    while (grp + 1 < p.n_groups && int(blockIdx.x) >= p.cta_begin[grp + 1]) ++grp;
    const int in_group = blockIdx.x - p.cta_begin[grp];
    pair = in_group / p.ctas_per_pair[grp];
    part = (in_group - pair * p.ctas_per_pair[grp]) % p.parts[grp];
    jt = (in_group - pair * p.ctas_per_pair[grp]) / p.parts[grp];
    for (;; ++win) {
      const int vis = p.causal ? min(n_jt, ((win + 1) * p.window[grp] * BQ2 + BT - 1) / BT) : n_jt;
      if (jt < vis) break;
      jt -= vis;
    }
  }
  const int parts = p.parts[grp];
  const int window = p.window[grp];
  const int slot0 = p.first_slot[grp];
  const int n_layers = p.first_slot[grp + 1] - slot0;
  const int hk = pair % p.Hkv;
  const int b = pair / p.Hkv;
  const int G = p.Hq / p.Hkv;
  const int kv0 = jt * BT;
  const int qt_first = max(p.causal ? (kv0 / BQ2) : 0, win * window);
  const int per_stream = min(n_qt, (win + 1) * window) - qt_first;
  const int n_streams = n_layers * G;
  const int stream0 = part * n_streams / parts;
  const int n_iter = ((part + 1) * n_streams / parts - stream0) * per_stream;

  auto decode_iter = [&](int it, int& li, int& hq, int& q0) {
    const int stream = it / per_stream;
    const int qi = it - stream * per_stream;
    li = (stream0 + stream) / G;
    hq = hk * G + (stream0 + stream - li * G);
    q0 = (qt_first + qi) * BQ2;
  };
  auto load_step = [&](int it, uint32_t leader) {
    int li, hq, q0;
    decode_iter(it, li, hq, q0);
    const int s = it % L::STAGES;
    mbar_expect_tx_e(&q_full[s], L::STAGE, leader);
    uint8_t* dst = smem + L::OFF_RING + s * L::STAGE;
#pragma unroll
    for (int h = 0; h < HALVES; ++h) {
      tma_load_4d_e(dst + h * QHALF_BYTES, &p.map_q[slot0 + li], &q_full[s], h * 64, hq, q0, b, leader);
      tma_load_4d_e(dst + L::Q_TILE + h * QHALF_BYTES, &p.map_do[slot0 + li], &q_full[s], h * 64, hq, q0, b, leader);
    }
  };

  // The loads that everything waits for go out before the block has set itself up: the TMA warp initialises the barriers
  // and fills the ring, then the block meets.
  if (warp == 0) {
    const uint32_t leader = elect_one();
    if (leader) {
      mbar_init(kv_full, 1);
      for (int s = 0; s < L::STAGES; ++s) {
        mbar_init(&q_full[s], 1 + 64);
        mbar_init(&q_empty[s], 1);
      }
      for (int i = 0; i < 2; ++i) {
        mbar_init(&st_full[i], 1);
        mbar_init(&dp_free[i], L::STEP_THREADS);
        mbar_init(&pds_ready[i], L::STEP_THREADS);
      }
      for (int i = 0; i < 2; ++i) mbar_init(&dq_full[i], 1);
      mbar_init(dq_free, 128);
      mbar_init(acc_done, 1);
      mbar_init(a_ready, 256);
      mbar_fence_init();
      fence_proxy_async_smem();
    }
    __syncwarp();
    grid_dep_wait();
    mbar_expect_tx_e(kv_full, 2 * L::KV_TILE, leader);
#pragma unroll
    for (int h = 0; h < HALVES; ++h) {
      tma_load_4d_e(smem + L::OFF_K + h * HALF_BYTES, &p.map_k[grp], kv_full, h * 64, hk, kv0, b, leader);
      tma_load_4d_e(smem + L::OFF_V + h * HALF_BYTES, &p.map_v[grp], kv_full, h * 64, hk, kv0, b, leader);
    }
    for (int it = 0; it < min(n_iter, L::STAGES); ++it) load_step(it, leader);
  }
  // constant operand tiles: ones in the first three columns, and the zeros
  if (threadIdx.x < 256) {
    const bool ones = threadIdx.x < 128;   // row i, columns 0-7 = 1,1,1,0,0,0,0,0
    *reinterpret_cast<uint4*>(smem + (ones ? L::OFF_ONES : L::OFF_ZERO) + (threadIdx.x & 127) * 16) =
        make_uint4(ones ? 0x3F803F80u : 0u, ones ? 0x00003F80u : 0u, 0u, 0u);
  }
  fence_proxy_async_smem();
  if (warp == 1) {
    tmem_alloc(tmem_slot, 512);
    tmem_relinquish();
  }
  tc_fence_before_sync();
  __syncthreads();
  tc_fence_after_sync();
  const uint32_t tmem_base = *tmem_slot;
  grid_dep_wait();
  const uint32_t tm_dp = tmem_base + 128;                                   // [2] at DH 64
  const uint32_t tm_dq = tmem_base + (L::SMALL ? 256 : 192);
  const uint32_t tm_dk = tm_dq + 64;
  const uint32_t tm_dv = tm_dk + DH;
  const uint32_t tm_k = tmem_base + 448, tm_v = tmem_base + 480;            // DH 64

  if (warp == 0) {
    // ------------------------------ TMA producer ------------------------------
    const uint32_t leader = elect_one();  // the whole warp runs the loop; one lane issues
    for (int it = L::STAGES; it < n_iter; ++it) {
      if (!mbar_wait(&q_empty[it % L::STAGES], ((it / L::STAGES) & 1) ^ 1, err)) break;
      load_step(it, leader);
    }
    grid_dep_launch();   // all loads are out
  } else if (warp == 1) {
    // ------------------------------ MMA issuer ------------------------------
    {
      const uint32_t leader = elect_one();  // the whole warp runs the loop; one lane issues
      constexpr uint32_t idesc_st = umma_idesc_bf16(BT, BQ2, 0, 0);   // [128 keys x 64 queries]
      constexpr uint32_t idesc_acc = umma_idesc_bf16(BT, DH, 0, 1);   // A from TMEM, B MN-major
      // dQ^T [dh x 64 queries] = K^T dS^T, both operands MN-major.  The instruction always spans 128 rows; with
      // DH == 64 the upper 64 are fed from the V tile that follows K in shared memory and are never read.
      constexpr uint32_t idesc_dq = umma_idesc_bf16(128, BQ2, 1, 1);
      constexpr uint32_t hi = desc_hi_sw128(1024);
      constexpr uint32_t hi_plain = desc_hi_plain(128);
      // low descriptor words of the resident tiles; per MMA only a constant is added
      const uint32_t k_lo = desc_lo_sw128(smem_u32(smem + L::OFF_K), 0);
      const uint32_t v_lo = desc_lo_sw128(smem_u32(smem + L::OFF_V), 0);
      const uint32_t kmn_lo = desc_lo_sw128(smem_u32(smem + L::OFF_K), HALF_BYTES);   // K as MN-major A
      const uint32_t ds_lo = desc_lo_sw128(smem_u32(smem + L::OFF_DS), 0);            // dS^T as MN-major B
      // 16-column K-major tiles whose columns 8-15 are all zero share one block of zeros: the leading-dimension
      // offset of each descriptor is the distance from the tile's first half to that block
      const uint32_t zero_addr = smem_u32(smem + L::OFF_ZERO);
      const uint32_t ones_lo = desc_lo_plain(smem_u32(smem + L::OFF_ONES), zero_addr - smem_u32(smem + L::OFF_ONES));
      const uint32_t stat_base = smem_u32(smem + L::OFF_STAT);
      const uint32_t ring = smem_u32(smem + L::OFF_RING);
      bool ok = mbar_wait(kv_full, 0, err);
      if (L::SMALL && ok) ok = mbar_wait(a_ready, 0, err);
      // One score product and the statistics of its queries: S^T - LSE / scale, dP^T - Delta.
      auto product = [&](uint32_t d, uint32_t a_tmem, uint32_t a_lo, uint32_t b_lo, uint32_t stat_addr) {
#pragma unroll
        for (int ks = 0; ks < KSTEPS_DH; ++ks) {
          const uint32_t b = desc_lo_add(b_lo, (ks / 4) * QHALF_BYTES + (ks % 4) * 32);
          if constexpr (L::SMALL) umma_ts_w(d, a_tmem + ks * 8, b, hi, idesc_st, ks != 0, leader);
          else umma_ss_w(d, desc_lo_add(a_lo, (ks / 4) * HALF_BYTES + (ks % 4) * 32), b, hi, idesc_st, ks != 0, leader);
        }
        umma_ss_w(d, ones_lo, desc_lo_plain(stat_addr, zero_addr - stat_addr), hi_plain, idesc_st, 1, leader);
      };
      auto issue_s = [&](int it) {
        const int s = it % L::STAGES;
        product(tmem_base + (it & 1) * 64, tm_k, k_lo, desc_lo_sw128(ring + s * L::STAGE, 0), stat_base + s * STAT_BYTES);
      };
      auto issue_dp = [&](int it) {
        const int s = it % L::STAGES;
        product(tm_dp + (L::SMALL ? (it & 1) * 64 : 0), tm_v, v_lo, desc_lo_sw128(ring + s * L::STAGE + L::Q_TILE, 0),
                stat_base + s * STAT_BYTES + BQ2 * 16);
      };
      auto stage_full = [&](int it) -> bool {
        const bool w = mbar_wait(&q_full[it % L::STAGES], (it / L::STAGES) & 1, err);
        tc_fence_after_sync();
        return w;
      };
      // DH 128.  The single dP^T buffer takes the next step once the compute warps hold the previous one in registers.
      auto issue_scores = [&](int it) -> bool {
        if (!stage_full(it)) return false;
        issue_s(it);
        if (it > 0 && !mbar_wait(&dp_free[(it - 1) & 1], ((it - 1) >> 1) & 1, err)) return false;
        tc_fence_after_sync();
        issue_dp(it);
        umma_commit(&st_full[it & 1], leader);
        return true;
      };
      if constexpr (L::SMALL) {
        for (int it = 0; it < min(n_iter, 2) && ok; ++it) {
          ok = stage_full(it);
          if (!ok) break;
          issue_s(it);
          issue_dp(it);
          umma_commit(&st_full[it], leader);
        }
      } else {
        if (ok && n_iter > 0) ok = issue_scores(0);
      }
      for (int it = 0; it < n_iter && ok; ++it) {
        // DH 128: S^T of the next step goes to the other score buffer; its previous readers (the accumulate MMAs
        // of step it-1) precede this in the in-order tensor pipe
        if constexpr (L::SMALL) {
          // dP^T of the step after the next, over the buffer that this step's warps have read
          if (it + 2 < n_iter) {
            if (!stage_full(it + 2) || !mbar_wait(&dp_free[it & 1], (it >> 1) & 1, err)) { ok = false; break; }
            tc_fence_after_sync();
            issue_dp(it + 2);
          }
        } else {
          if (it + 1 < n_iter && !issue_scores(it + 1)) { ok = false; break; }
        }
        if (!mbar_wait(&pds_ready[it & 1], (it >> 1) & 1, err)) { ok = false; break; }
        tc_fence_after_sync();
        const int s = it % L::STAGES;
        const uint32_t qmn_lo = desc_lo_sw128(ring + s * L::STAGE, QHALF_BYTES);                 // Q  as MN-major B
        const uint32_t domn_lo = desc_lo_sw128(ring + s * L::STAGE + L::Q_TILE, QHALF_BYTES);    // dO as MN-major B
        const uint32_t tm = tmem_base + (it & 1) * 64;
        // P^T of queries [32w, 32w+32) sits in 32-bit columns [32w, 32w+16) of the score buffer, dS^T in [32w+16, 32w+32)
#pragma unroll
        for (int ks = 0; ks < KSTEPS_Q; ++ks)  // dV += P^T dO
          umma_ts_w(tm_dv, tm + (ks / 2) * 32 + (ks % 2) * 8, desc_lo_add(domn_lo, ks * 2048), hi, idesc_acc, (it | ks) != 0, leader);
#pragma unroll
        for (int ks = 0; ks < KSTEPS_Q; ++ks)  // dK += dS^T Q
          umma_ts_w(tm_dk, tm + (ks / 2) * 32 + 16 + (ks % 2) * 8, desc_lo_add(qmn_lo, ks * 2048), hi, idesc_acc, (it | ks) != 0, leader);
        umma_commit(&q_empty[s], leader);  // the ring stage is free as soon as dV and dK have read it
        // DH 64: S^T of the step after the next, over the score buffer that dV and dK have just read, goes ahead of dQ^T, whose
        // dS^T tile has a twin
        if (L::SMALL && it + 2 < n_iter) {
          issue_s(it + 2);
          umma_commit(&st_full[it & 1], leader);
        }
        if (it > 0 && !mbar_wait(dq_free, (it - 1) & 1, err)) { ok = false; break; }
        tc_fence_after_sync();
#pragma unroll
        for (int ks = 0; ks < KSTEPS_KV; ++ks)  // dQ^T = K^T dS^T
          umma_ss_w(tm_dq, desc_lo_add(kmn_lo, ks * 2048), desc_lo_add(ds_lo, (it & (L::DS_BUFS - 1)) * (BT * BQ2 * 2) + ks * 2048), hi, idesc_dq, ks != 0, leader);
        umma_commit(&dq_full[it & 1], leader);
      }
      if (ok) umma_commit(acc_done, leader);
    }
  } else if (warp < 10) {
    // ------------------------------ compute warpgroups ------------------------------
    const int wg = (warp - 2) >> 2;     // DH 128: query columns [wg*32, wg*32+32) of every step; 64: all of every other step
    const int quarter = warp & 3;       // TMEM lane quarter of this warp
    const int r = quarter * 32 + lane;  // key row inside the tile == TMEM lane
    const uint32_t lane_sel = uint32_t(quarter * 32) << 16;
    const int kv_row = kv0 + r;
    const uint64_t c2 = pack_f2(p.scale_log2, p.scale_log2);
    uint8_t* ds_smem = smem + L::OFF_DS;
    if constexpr (L::SMALL) {   // K (warpgroup 0) and V (warpgroup 1) as A operands in TMEM, key row by key row
      bool w = mbar_wait(kv_full, 0, err);
      if (__all_sync(0xffffffffu, w)) {
        uint32_t row[32];
#pragma unroll
        for (int j = 0; j < 8; ++j) {
          const uint4 v = *reinterpret_cast<const uint4*>(smem + (wg == 0 ? L::OFF_K : L::OFF_V) + sw128_offset(r, j));
          row[4 * j] = v.x;
          row[4 * j + 1] = v.y;
          row[4 * j + 2] = v.z;
          row[4 * j + 3] = v.w;
        }
        tmem_st_x32((wg == 0 ? tm_k : tm_v) + lane_sel, row);
        tmem_st_wait();
        tc_fence_before_sync();
        mbar_arrive(a_ready);
      }
    }
    // DH 128: the warpgroups take half of the queries of every step each.  DH 64, where a step has half the MMA time and the
    // same exponentials: every other step each, so that the loads, stores and waits of one fall into the exponentials of the
    // other.
    constexpr int STRIDE = L::SMALL ? 2 : 1, PARTS = L::SMALL ? 2 : 1;
    int qi = L::SMALL ? wg % per_stream : 0;  // query tile index of the current step inside its stream
    bool ok = true;
    for (int it = L::SMALL ? wg : 0; it < n_iter; it += STRIDE) {
      const int set = it & 1;
      ok = mbar_wait(&st_full[set], (it >> 1) & 1, err);
      if (!__all_sync(0xffffffffu, ok)) { ok = false; break; }
      tc_fence_after_sync();
      const int q0 = (qt_first + qi) * BQ2;
      const bool diag = p.causal && q0 < kv0 + BT;                    // the query tile straddles the diagonal
      uint8_t* const ds_tile = ds_smem + (it & (L::DS_BUFS - 1)) * (BT * BQ2 * 2);
#pragma unroll
      for (int part = 0; part < PARTS; ++part) {
        // P^T and dS^T (bf16 pairs) overwrite the 32 score columns they come from, which no other thread reads: P^T the
        // first 16, dS^T the others
        const int half = L::SMALL ? part : wg;                        // queries [32 half, 32 half + 32)
        const uint32_t col = tmem_base + set * 64 + half * 32 + lane_sel;
        uint32_t st[32], dp[32];
        tmem_ld_x32(col, st);
        tmem_ld_x32(tm_dp + (L::SMALL ? set * 64 : 0) + half * 32 + lane_sel, dp);
        const int first_visible = diag ? kv_row - q0 - half * 32 : 0; // columns below this are masked for this key row
        uint32_t pk[16], dk[16];
        tmem_ld_wait();
        if (part == PARTS - 1) {
          tc_fence_before_sync();
          mbar_arrive(&dp_free[set]);
        }
#pragma unroll
        for (int i = 0; i < 16; ++i) {
          const uint64_t x = fmul2(pack_f2(__uint_as_float(st[2 * i]), __uint_as_float(st[2 * i + 1])), c2);
          float e0 = fast_exp2(f2_lo(x)), e1 = fast_exp2(f2_hi(x));
          if (diag) {
            e0 = 2 * i < first_visible ? 0.f : e0;
            e1 = 2 * i + 1 < first_visible ? 0.f : e1;
          }
          pk[i] = pack_bf16(e0, e1);
          const uint64_t d = fmul2(pack_f2(e0, e1), pack_f2(__uint_as_float(dp[2 * i]), __uint_as_float(dp[2 * i + 1])));
          dk[i] = pack_bf16(f2_lo(d), f2_hi(d));
        }
        // keys beyond the sequence contribute nothing (their K/V rows are zero-filled; dK/dV rows are not stored)
        tmem_st_x16(col, pk);
        tmem_st_x16(col + 16, dk);
        // dS^T also goes to shared memory as the B operand of dQ^T = K^T dS^T; the product of the step that last used the
        // tile must have finished reading it
        if (part == 0 && it >= L::DS_BUFS) {
          ok = mbar_wait(&dq_full[(it - L::DS_BUFS) & 1], ((it - L::DS_BUFS) >> 1) & 1, err);
          if (!__all_sync(0xffffffffu, ok)) { ok = false; break; }
        }
#pragma unroll
        for (int j = 0; j < 4; ++j)
          *reinterpret_cast<uint4*>(ds_tile + sw128_offset(r, half * 4 + j)) =
              make_uint4(dk[4 * j], dk[4 * j + 1], dk[4 * j + 2], dk[4 * j + 3]);
      }
      if (!ok) break;
      tmem_st_wait();
      fence_proxy_async_smem();  // dS^T is read by the tensor core's proxy
      tc_fence_before_sync();
      mbar_arrive(&pds_ready[set]);
      qi += STRIDE;
      while (qi >= per_stream) qi -= per_stream;
    }
    ok = __all_sync(0xffffffffu, ok);
    if (ok) {
      bool w = mbar_wait(acc_done, 0, err);
      ok = __all_sync(0xffffffffu, w);
    }
    if (ok) {
      tc_fence_after_sync();
      // Warpgroup 0 adds dK (scaled), warpgroup 1 adds dV: each warp moves its 32 rows, 32 columns at a time, into
      // shared memory that the finished MMAs have left (dK over the ring, dV over K and V) and adds them with one TMA
      // reduction each, which clips rows beyond the sequence.  (Adding straight from registers, one 16-byte piece of
      // 32 different rows per instruction, moves one line per cycle: with the early loads above, a CTA of dh 128 spends
      // 7 us besides its steps instead of 12, at 1.25 us a step.)
      const uint32_t src = (wg == 0 ? tm_dk : tm_dv) + lane_sel;
      const float mul = wg == 0 ? p.scale : 1.f;
      uint8_t* area = smem + (wg == 0 ? L::OFF_RING : L::OFF_K) + quarter * 4096;
      const CUtensorMap* map = wg == 0 ? &p.map_dk[grp] : &p.map_dv[grp];
      if (kv0 + quarter * 32 < p.S) {
#pragma unroll 1
        for (int c = 0; c < DH / 32; ++c) {
          uint32_t a[32];
          tmem_ld_x32(src + c * 32, a);
          tmem_ld_wait();
          uint8_t* tile = area + c * HALF_BYTES;
#pragma unroll
          for (int v4 = 0; v4 < 8; ++v4)
            *reinterpret_cast<float4*>(tile + sw128_offset(lane, v4)) =
                make_float4(__uint_as_float(a[4 * v4]) * mul, __uint_as_float(a[4 * v4 + 1]) * mul,
                            __uint_as_float(a[4 * v4 + 2]) * mul, __uint_as_float(a[4 * v4 + 3]) * mul);
          fence_proxy_async_smem();
          __syncwarp();
          if (lane == 0) {
            tma_reduce_add_4d(map, tile, c * 32, hk, kv0 + quarter * 32, b);
            asm volatile("cp.async.bulk.commit_group;" ::: "memory");
          }
        }
        if (lane == 0) asm volatile("cp.async.bulk.wait_group.read 0;" ::: "memory");
        __syncwarp();
      }
    }
  } else if (warp >= 14) {
    // ------------------------------ statistics ------------------------------
    // Thread t forms the two operand rows of query column t, -LSE / scale and -Delta in three bf16 terms each, in the ring slot
    // of the step, from values that it asked for two steps before.  (As a side job of the drain warpgroup they took 500 to 600
    // of its 1800 cycles a step.)
    const int t = int(threadIdx.x) - 14 * 32;
    const float lse_mul = -1.f / p.scale;
    uint8_t* const row = smem + L::OFF_STAT + t * 16;
    int li = stream0 / G, g = stream0 % G, qi = 0, asked = 0;
    auto ask = [&](float& lse, float& delta) {   // of the next step; a query beyond the sequence: exp2 underflows to zero
      const int q = (qt_first + qi) * BQ2 + t;
      lse = 30000.f * p.scale;
      delta = 0.f;
      if (asked < n_iter && q < p.S) {
        const size_t at = (size_t(b) * p.Hq + hk * G + g) * p.S + q;
        lse = p.lse[slot0 + li][at];
        delta = p.delta[slot0 + li][at];
      }
      ++asked;
      if (++qi == per_stream) {
        qi = 0;
        if (++g == G) {
          g = 0;
          ++li;
        }
      }
    };
    float l0, d0, l1, d1, l2, d2;
    ask(l0, d0);
    ask(l1, d1);
    int s = 0;
    uint32_t ph = 1;
    for (int it = 0; it < n_iter; ++it) {
      ask(l2, d2);
      const bool ok = mbar_wait(&q_empty[s], ph, err);
      if (!__all_sync(0xffffffffu, ok)) break;
      *reinterpret_cast<uint4*>(row + s * STAT_BYTES) = split3_bf16(l0 * lse_mul);
      *reinterpret_cast<uint4*>(row + s * STAT_BYTES + BQ2 * 16) = split3_bf16(-d0);
      fence_proxy_async_smem();
      mbar_arrive(&q_full[s]);
      l0 = l1;
      d0 = d1;
      l1 = l2;
      d1 = d2;
      if (++s == L::STAGES) {
        s = 0;
        ph ^= 1;
      }
    }
  } else {
    // ------------------------------ dQ drain warpgroup ------------------------------
    // TMEM lane == column of dQ (dh index): this warp owns dh columns [32*quarter, 32*quarter + 32) of the
    // step's 64 queries, lays them out as [16 groups of four queries][32 columns][4] fp32 in shared memory, a lane's four
    // queries with one store, and adds them to the accumulator with one 8 KB bulk reduction.
    // The chain of a step is short on purpose: dQ^T to registers, dq_free, the copy.  Stored a float at a time, and with the
    // operand tiles of the statistics formed here too, ahead of dq_free, this warpgroup was busy for 1650 of a step's 1830
    // cycles at DH 64 (1720 of 2020 at 128) and the step waited for it.
    const int quarter = warp & 3;
    const uint32_t lane_sel = uint32_t(quarter * 32) << 16;
    const bool active = quarter * 32 < DH;  // with DH == 64 the upper lanes hold nothing
    // the reduction of the step before (with the idle warps' space at DH 64, of the step before that) has a step to read its buffer
    constexpr int BUFS = L::DQ_BUFS;
    uint8_t* const stg = smem + L::OFF_DQ + quarter * BUFS * DQ_STAGE_BYTES;
    int li = stream0 / G, g = stream0 % G, qi = 0;
    bool ok = true;
    for (int it = 0; it < n_iter; ++it) {
      ok = mbar_wait(&dq_full[it & 1], (it >> 1) & 1, err);
      if (!__all_sync(0xffffffffu, ok)) { ok = false; break; }
      tc_fence_after_sync();
      uint32_t a[64];
      if (active) {
        tmem_ld_x32(tm_dq + lane_sel, *reinterpret_cast<uint32_t(*)[32]>(&a[0]));
        tmem_ld_x32(tm_dq + lane_sel + 32, *reinterpret_cast<uint32_t(*)[32]>(&a[32]));
        tmem_ld_wait();
      }
      tc_fence_before_sync();
      mbar_arrive(dq_free);
      if (active && p.dq_direct) {
        // One key tile: the partial is the whole sum, and goes out as dQ: rounded, a lane's eight queries a row of 16 bytes of an
        // 8x8 matrix in shared memory, back transposed as eight columns of one query, 16 bytes a store.  (Exchanged between lanes
        // instead it took 1900 cycles a step, more than the rest of the step.)
        const int q0 = (qt_first + qi) * BQ2 + lane / 4;
        const size_t at = ((size_t(b) * p.S + q0) * p.Hq + hk * G + g) * DH + quarter * 32 + lane % 4 * 8, step = size_t(8) * p.Hq * DH;
        void* const dq = p.dq[slot0 + li];
        // column c of an eight of queries at place (c ^ 2 (c / 8)), which keeps both the stores and the matrices' rows clear of
        // bank conflicts; row i of matrix m: column 8 (i / 2) + 2 m + i % 2, so that a lane's four registers are adjacent columns
        auto place = [](int c) { return uint32_t(c ^ (c >> 3 << 1)) * 16; };
        uint8_t* const put = stg + place(lane);
        const uint32_t get = smem_u32(stg) + place((lane & 6) * 4 + (lane >> 3) * 2 + (lane & 1));
        __syncwarp();   // (the reads of the step before)
#pragma unroll
        for (int e = 0; e < 8; ++e) {
          auto pair = [&](int i) { return pack_bf16(__uint_as_float(a[8 * e + i]) * p.scale, __uint_as_float(a[8 * e + i + 1]) * p.scale); };
          *reinterpret_cast<uint4*>(put + e * 512) = make_uint4(pair(0), pair(2), pair(4), pair(6));
        }
        __syncwarp();
#pragma unroll
        for (int e = 0; e < 8; ++e) {
          uint4 v;
          ldsm_x4_t(get + e * 512, v.x, v.y, v.z, v.w);
          if (q0 + 8 * e < p.S) store_dq(dq, p.dq_f32, at + e * step, v);
        }
      } else if (active) {
        const size_t tile = ((size_t(b) * p.Hq + hk * G + g) * n_qt + (qt_first + qi)) * (DH / 32) + quarter;
        float* dst = p.dq_acc[slot0 + li] + tile * (BQ2 * 32);
        uint8_t* const buf = stg + (it & (BUFS - 1)) * DQ_STAGE_BYTES;
        // the reduction that last used the buffer has read it
        if (lane == 0) asm volatile("cp.async.bulk.wait_group.read %0;" ::"n"(BUFS - 1) : "memory");
        __syncwarp();
#pragma unroll
        for (int q = 0; q < BQ2; q += 4) *reinterpret_cast<uint4*>(buf + q * 128 + lane * 16) = make_uint4(a[q], a[q + 1], a[q + 2], a[q + 3]);
        fence_proxy_async_smem();
        __syncwarp();
        if (lane == 0) {
          asm volatile("cp.reduce.async.bulk.global.shared::cta.bulk_group.add.f32 [%0], [%1], %2;" ::"l"(dst), "r"(smem_u32(buf)),
                       "n"(DQ_STAGE_BYTES)
                       : "memory");
          asm volatile("cp.async.bulk.commit_group;" ::: "memory");
        }
      }
      if (++qi == per_stream) {
        qi = 0;
        if (++g == G) {
          g = 0;
          ++li;
        }
      }
    }
    // the reductions must have read the block's shared memory before it goes away (their writes complete with the grid)
    if (lane == 0) asm volatile("cp.async.bulk.wait_group.read 0;" ::: "memory");
    __syncwarp();
  }

  tc_fence_before_sync();
  __syncthreads();
  if (warp == 1) {
    tc_fence_after_sync();
    tmem_dealloc(tmem_base, 512);
  }
}

// The passes before and after bwd_kernel, each ONE launch for all member layers of a bwd_kernel launch (blockIdx.y is
// the layer's slot): a layer's share is a few microseconds at small sizes, where every launch cost as much again
// (Delta, clears and conversion of three layers of 3 x 776 tokens: 11 launches, 39 us -> 2 launches, 20 us).
struct AuxParams {
  const __nv_bfloat16* o[MAX_GROUP];
  const __nv_bfloat16* d_o[MAX_GROUP];
  void* dq[MAX_GROUP];        // bf16 or (dq_f32) the bf16 values as fp32
  float* delta[MAX_GROUP];
  float* dq_acc[MAX_GROUP];
  float* dk_sum[MAX_GROUP];   // per group
  float* dv_sum[MAX_GROUP];
  int n_groups;
  int dq_f32;
  int B, S, Hq;
  size_t acc_v4;              // 16-byte pieces of one dQ accumulator
  size_t kv_v4;               // 16-byte pieces of one dK (dV) sum
  float scale;
};

// After: dq[b,s,hq,:] = bf16(scale * accumulator), from the blocked fp32 layout [b][hq][tile][quarter][16][32 columns][4 queries].
// A warp takes 16 queries x 32 columns at a time: a lane loads its column's queries, four of them with each of four 16-byte
// loads, and three exchanges (lanes 1, 2 and 4 apart) leave it with eight consecutive columns of two queries.  Bound: HBM.
template <int DH>
__global__ void dq_convert_kernel(const __grid_constant__ AuxParams p) {
  grid_dep_wait();
  const float4* acc = reinterpret_cast<const float4*>(p.dq_acc[blockIdx.y]);
  const int S = p.S, Hq = p.Hq, lane = threadIdx.x & 31;
  const float scale = p.scale;
  const int n_qt = (S + BQ2 - 1) / BQ2;
  const size_t units = size_t(p.B) * Hq * n_qt * (DH / 32) * (BQ2 / 16);
  const size_t stride = size_t(gridDim.x) * blockDim.x / 32;
  const bool b0 = lane & 1, b1 = lane & 2, b2 = lane & 4;
  const int own = (b0 ? 4 : 0) + (b1 ? 2 : 0) + (b2 ? 1 : 0);   // of eight queries, the one this lane stores
  for (size_t u = (size_t(blockIdx.x) * blockDim.x + threadIdx.x) / 32; u < units; u += stride) {
    if (u + stride >= units) grid_dep_launch();
    const size_t block = u / (BQ2 / 16);                        // tile * (DH / 32) + quarter
    const size_t tile = block / (DH / 32);                      // (b * Hq + hq) * n_qt + qt
    const size_t bh = tile / n_qt;
    const int s0 = int(tile % n_qt) * BQ2 + int(u % (BQ2 / 16)) * 16;
    if (s0 >= S) continue;
    float4 f[4];
#pragma unroll
    for (int i = 0; i < 4; ++i) f[i] = acc[u * 128 + i * 32 + lane];
    const int hq = int(bh % Hq), bb = int(bh / Hq);
    const int col = int(block % (DH / 32)) * 32 + (lane & 24);
#pragma unroll
    for (int h = 0; h < 2; ++h) {
      const float4 x = f[2 * h], y = f[2 * h + 1];
      const uint32_t w[4] = {pack_bf16(x.x * scale, x.y * scale), pack_bf16(x.z * scale, x.w * scale),   // queries 0 1, 2 3,
                             pack_bf16(y.x * scale, y.y * scale), pack_bf16(y.z * scale, y.w * scale)};  // 4 5, 6 7
      const uint32_t e0 = __shfl_xor_sync(0xffffffffu, b0 ? w[0] : w[2], 1), e1 = __shfl_xor_sync(0xffffffffu, b0 ? w[1] : w[3], 1);
      const uint32_t lo0 = b0 ? e0 : w[0], lo1 = b0 ? e1 : w[1], hi0 = b0 ? w[2] : e0, hi1 = b0 ? w[3] : e1;
      // two columns of four queries
      const uint32_t t0 = __byte_perm(lo0, hi0, 0x5410), t1 = __byte_perm(lo0, hi0, 0x7632);
      const uint32_t t2 = __byte_perm(lo1, hi1, 0x5410), t3 = __byte_perm(lo1, hi1, 0x7632);
      const uint32_t g0 = __shfl_xor_sync(0xffffffffu, b1 ? t0 : t2, 2), g1 = __shfl_xor_sync(0xffffffffu, b1 ? t1 : t3, 2);
      // four columns of two queries: (x0, y0) and (x1, y1)
      const uint32_t x0 = b1 ? g0 : t0, y0 = b1 ? t2 : g0, x1 = b1 ? g1 : t1, y1 = b1 ? t3 : g1;
      const uint32_t k0 = __shfl_xor_sync(0xffffffffu, b2 ? x0 : x1, 4), k1 = __shfl_xor_sync(0xffffffffu, b2 ? y0 : y1, 4);
      const uint4 v = b2 ? make_uint4(k0, k1, x1, y1) : make_uint4(x0, y0, k0, k1);
      const int s = s0 + h * 8 + own;
      if (s >= S) continue;
      const size_t at = ((size_t(bb) * S + s) * Hq + hq) * DH + col;
      store_dq(p.dq[blockIdx.y], p.dq_f32, at, v);
    }
  }
}

// fp32 interface: the pre-pass reads the caller's O and dO, stores dO as bf16 (to d_o), and beside the slots rounds a list of
// other tensors; a launch of its own for that took 3 us of the smallest steps' 42.
template <bool F32>
struct PrepareParams : AuxParams {};
template <>
struct PrepareParams<true> : AuxParams {
  const float *o32[MAX_GROUP], *do32[MAX_GROUP];
  int cast_rows;              // blockIdx.y beyond the slots: round the list
  CastParams casts;
};

// Before: clears the slot's dQ accumulator and the slot's share of the dK / dV sums (stores, nothing waits for them),
// and forms Delta[b,hq,s] = sum_c dO[b,s,hq,c] * O[b,s,hq,c].
// A row of DH bf16 is DH/8 16-byte pieces, and a load of a warp takes 256/DH rows (every lane busy): of consecutive tokens of one
// head, whose results lie side by side, with the other heads of these tokens in the warps beside it.  Two such loads of
// O and of dO are in flight, reduced inside the DH/8-lane segments.  Bound: HBM.
template <int DH, bool F32>
__global__ void bwd_prepare_kernel(const __grid_constant__ PrepareParams<F32> p) {
  constexpr int LANES = DH / 8;          // lanes per row
  constexpr int ROWS = 32 / LANES;       // rows per warp and load
  grid_dep_wait();
  const int slot = blockIdx.y;
  if constexpr (F32) {
    const int slots = gridDim.y - p.cast_rows;
    if (slot >= slots) {
      cast_chunks(p.casts, (slot - slots) * gridDim.x + blockIdx.x, p.cast_rows * gridDim.x);
      return;
    }
  }
  const size_t first = size_t(blockIdx.x) * blockDim.x + threadIdx.x, stride = size_t(gridDim.x) * blockDim.x;
  auto clear = [&](float* dst, size_t n) {
    float4* d = reinterpret_cast<float4*>(dst);
    for (size_t i = first; i < n; i += stride) d[i] = make_float4(0.f, 0.f, 0.f, 0.f);
  };
  clear(p.dq_acc[slot], p.acc_v4);
  if (slot < p.n_groups) {
    clear(p.dk_sum[slot], p.kv_v4);
    clear(p.dv_sum[slot], p.kv_v4);
  }
  const __nv_bfloat16* o = p.o[slot];
  const __nv_bfloat16* d_o = p.d_o[slot];
  float* const delta = p.delta[slot];
  const int S = p.S, Hq = p.Hq;
  constexpr int TOKS = 2 * ROWS;         // of a unit
  const int per_seq = (S + TOKS - 1) / TOKS;
  const size_t units = size_t(p.B) * per_seq * Hq;
  const int lane = threadIdx.x & 31;
  const int sub = lane / LANES, piece = lane % LANES;
  auto dot8 = [](const uint4& a, const uint4& g) {
    const __nv_bfloat162* pa = reinterpret_cast<const __nv_bfloat162*>(&a);
    const __nv_bfloat162* pg = reinterpret_cast<const __nv_bfloat162*>(&g);
    float acc = 0.f;
#pragma unroll
    for (int i = 0; i < 4; ++i) {
      const float2 fa = __bfloat1622float2(pa[i]), fg = __bfloat1622float2(pg[i]);
      acc += fa.x * fg.x + fa.y * fg.y;
    }
    return acc;
  };
  for (size_t u = first >> 5; u < units; u += stride >> 5) {
    if (u + (stride >> 5) >= units) grid_dep_launch();
    const int hq = int(u % Hq);
    const size_t group = u / Hq, b = group / per_seq;
    const int s0 = int(group % per_seq) * TOKS + sub, s1 = s0 + ROWS;
    const size_t at = ((b * S + s0) * Hq + hq) * DH + piece * 8, next = size_t(ROWS) * Hq * DH;
    const uint4 z = make_uint4(0u, 0u, 0u, 0u);
    uint4 a0 = z, g0 = z, a1 = z, g1 = z;
    if constexpr (F32) {
      auto rounded = [](const float* src) {
        const float4 x = *reinterpret_cast<const float4*>(src), y = *reinterpret_cast<const float4*>(src + 4);
        return make_uint4(pack_bf16(x.x, x.y), pack_bf16(x.z, x.w), pack_bf16(y.x, y.y), pack_bf16(y.z, y.w));
      };
      __nv_bfloat16* const out = const_cast<__nv_bfloat16*>(d_o);
      if (s0 < S) {
        a0 = rounded(p.o32[slot] + at);
        g0 = rounded(p.do32[slot] + at);
        *reinterpret_cast<uint4*>(out + at) = g0;
      }
      if (s1 < S) {
        a1 = rounded(p.o32[slot] + at + next);
        g1 = rounded(p.do32[slot] + at + next);
        *reinterpret_cast<uint4*>(out + at + next) = g1;
      }
    } else {
      if (s0 < S) {
        a0 = *reinterpret_cast<const uint4*>(o + at);
        g0 = *reinterpret_cast<const uint4*>(d_o + at);
      }
      if (s1 < S) {
        a1 = *reinterpret_cast<const uint4*>(o + at + next);
        g1 = *reinterpret_cast<const uint4*>(d_o + at + next);
      }
    }
    float acc0 = dot8(a0, g0), acc1 = dot8(a1, g1);
#pragma unroll
    for (int sft = LANES / 2; sft > 0; sft >>= 1) {
      acc0 += __shfl_xor_sync(0xffffffffu, acc0, sft);
      acc1 += __shfl_xor_sync(0xffffffffu, acc1, sft);
    }
    // a lane each for the rows of the two loads
    const int s = piece == 0 ? s0 : s1;
    if (piece < 2 && s < S) delta[(b * Hq + hq) * S + s] = piece == 0 ? acc0 : acc1;
  }
}

int make_map_bshd(CUtensorMap* m, const void* base, int B, int S, int H, int dh, int rows) {
  uint64_t dims[4] = {uint64_t(dh), uint64_t(H), uint64_t(S), uint64_t(B)};
  uint64_t strides[3] = {uint64_t(dh) * 2, uint64_t(H) * dh * 2, uint64_t(S) * H * dh * 2};
  uint32_t box[4] = {64, 1, uint32_t(rows), 1};
  return make_tensor_map(m, base, 2, 4, dims, strides, box, true);
}

// fp32 [B,S,H,dh], boxes of 32 rows x 32 columns
int make_map_sum(CUtensorMap* m, const void* base, int B, int S, int H, int dh) {
  uint64_t dims[4] = {uint64_t(dh), uint64_t(H), uint64_t(S), uint64_t(B)};
  uint64_t strides[3] = {uint64_t(dh) * 4, uint64_t(H) * dh * 4, uint64_t(S) * H * dh * 4};
  uint32_t box[4] = {32, 1, 32, 1};
  return make_tensor_map(m, base, 4, 4, dims, strides, box, true);
}

size_t align256(size_t x) { return (x + 255) & ~size_t(255); }

// Orders the CTAs of a launch by their number of steps, longest first; 0 when there are more classes than the parameter
// block holds.  Three layers of 3 x 776 tokens, dh 64, cut as now, before heads of 64 had a pipeline of their own: 95 us in index
// order, 79 longest first.
int longest_first(BwdParams& p, int n_groups, int n_pairs, int n_jt, int n_qt, int G, int causal) {
  struct Class {
    int steps, ctas;
    uint32_t id;
  } cls[MAX_CLASSES];
  int n = 0, total = 0;
  for (int g = 0; g < n_groups; ++g) {
    const int streams = (p.first_slot[g + 1] - p.first_slot[g]) * G, w = p.window[g];
    for (int win = 0; win * w < n_qt; ++win) {
      const int vis = causal ? std::min(n_jt, ((win + 1) * w * BQ2 + BT - 1) / BT) : n_jt;
      for (int j = 0; j < vis; ++j) {
        if (n == MAX_CLASSES || win > 0xfff || j > 0xfff) return 0;
        const int tiles = std::min(n_qt, (win + 1) * w) - std::max(causal ? j * (BT / BQ2) : 0, win * w);
        cls[n++] = Class{tiles * streams / p.parts[g], n_pairs * p.parts[g], uint32_t(g) << 24 | uint32_t(win) << 12 | uint32_t(j)};
        total += n_pairs * p.parts[g];
      }
    }
  }
  if (total > 0xffff) return 0;
  std::stable_sort(cls, cls + n, [](const Class& a, const Class& b) { return a.steps > b.steps; });
  int end = 0;
  for (int c = 0; c < n; ++c) {
    end += cls[c].ctas;
    p.class_end[c] = uint16_t(end);
    p.class_id[c] = cls[c].id;
  }
  return n;
}

// Member layers of the launches' accumulators that are live at once: a launch takes whole donor groups until it
// holds MAX_GROUP member layers.
int max_layers_per_launch(const kvp_shape* s) { return s->L < MAX_GROUP ? s->L : MAX_GROUP; }

}  // namespace

int attn_bwd_read_status() {
  int v = 0;
  if (cudaMemcpyFromSymbol(&v, g_bwd_status, sizeof(int)) != cudaSuccess) return -1;
  if (v != 0) {
    int zero = 0;
    cudaMemcpyToSymbol(g_bwd_status, &zero, sizeof(int));
  }
  return v;
}

// Workspace: Delta [B,Hq,S] fp32 for every layer, then the fp32 dQ accumulators of the member layers of one launch
// (launches run one after the other and reuse them).
size_t attn_bwd_workspace(const kvp_shape* s, const int32_t* donor) {
  (void)donor;
  return size_t(s->L) * align256(size_t(s->B) * s->Hq * s->S * 4) +
         size_t(max_layers_per_launch(s)) * align256(dq_acc_floats(s->B, s->S, s->Hq, s->dh) * 4);
}

int attn_bwd_all(const kvp_shape* s, const int32_t* donor, int causal, float scale, const void* const* q,
                 const void* const* k, const void* const* v, const void* const* o, const void* const* d_o,
                 const float* const* lse, void* const* dq, const BwdF32* f32, bool dq_last, float* const* dk_sum, float* const* dv_sum, void* ws,
                 cudaStream_t stream) {
  const int dh = s->dh;
  const float sc = scale == 0.f ? 1.f / sqrtf(float(dh)) : scale;
  const size_t delta_bytes = align256(size_t(s->B) * s->Hq * s->S * 4);
  const size_t acc_bytes = align256(dq_acc_floats(s->B, s->S, s->Hq, dh) * 4);
  uint8_t* wsb = reinterpret_cast<uint8_t*>(ws);
  uint8_t* acc_base = wsb + size_t(s->L) * delta_bytes;
  if ((dh == 128 ? allow_smem<bwd_kernel<128>>(BwdSmem<128>::TOTAL) : allow_smem<bwd_kernel<64>>(BwdSmem<64>::TOTAL)) != cudaSuccess)
    return KVP_ERR_CUDA;

  // Donor groups, largest first; a launch takes groups until it holds MAX_GROUP member layers.  A launch writes
  // dK / dV of its donors through reductions into cleared buffers, so a donor shared by more than MAX_GROUP
  // layers is not supported.
  struct Group {
    int owner, n;
    int members[MAX_GROUP];
  };
  std::vector<Group> groups;
  for (int d = 0; d < s->L; ++d) {
    if (donor[d] != d) continue;
    Group g;
    g.owner = d;
    g.n = 0;
    for (int l = d; l < s->L; ++l)
      if (donor[l] == d) {
        if (g.n == MAX_GROUP) return KVP_ERR_UNSUPPORTED;
        g.members[g.n++] = l;
      }
    groups.push_back(g);
  }
  std::stable_sort(groups.begin(), groups.end(), [](const Group& a, const Group& b) { return a.n > b.n; });
  const int n_jt = (s->S + BT - 1) / BT, n_qt = (s->S + BQ2 - 1) / BQ2, n_pairs = s->Hkv * s->B;
  const int G = s->Hq / s->Hkv;
  const BwdSizes sizes{n_jt, n_qt, n_pairs, G, causal != 0, sm_count()};
  const double steps_per_sm = bwd_steps_per_sm(sizes, s->L);
  const int target = bwd_target_steps(steps_per_sm);
  size_t gi = 0;
  if (f32 != nullptr && f32->n_casts > MAX_CAST) {   // more than the pre-pass has room for
    const int rc = cast_tensors(f32->casts, f32->n_casts, stream);
    if (rc != KVP_OK) return rc;
  }
  // enough blocks for every slot to fill the device, no more than its pieces of 8 (16: convert) accumulators give work to
  const size_t acc_floats = dq_acc_floats(s->B, s->S, s->Hq, dh);
  auto aux_grid = [&](size_t per_thread, int slots) { return dim3(unsigned(min(size_t(sm_count()) * 16, (acc_floats / per_thread + 255) / 256)), slots); };
  // The pre-pass of the fp32 interface; the first of a call rounds the other tensors too.
  bool first_launch = true;
  auto prepare_f32 = [&](const AuxParams& ax, int slots, const float* const* o32, const float* const* do32) {
    PrepareParams<true> pre;
    static_cast<AuxParams&>(pre) = ax;
    std::copy(o32, o32 + slots, pre.o32);
    std::copy(do32, do32 + slots, pre.do32);
    pre.cast_rows = 0;
    dim3 grid = aux_grid(8, slots);
    if (first_launch && f32->n_casts <= MAX_CAST) {
      if (fill_casts(pre.casts, f32->casts, f32->n_casts) != f32->n_casts) return int(KVP_ERR_UNSUPPORTED);
      // About a block a chunk, up to eight blocks an SM.  (In one row of blocks, as many as a slot has, eight owners of 64 tokens took
      // 11.3 us instead of 7.6, of 2048 tokens, two heads, 79.3 instead of 73.4; ahead of the slots up to 0.8 us more.)
      const uint64_t rows = (uint64_t(pre.casts.chunks) + grid.x / 2) / grid.x;
      pre.cast_rows = int(std::max<uint64_t>(1, std::min<uint64_t>(rows, unsigned(sm_count()) * 8 / grid.x)));
      grid.y += pre.cast_rows;
    }
    first_launch = false;
    const cudaError_t e = launch_kernel(dh == 128 ? bwd_prepare_kernel<128, true> : bwd_prepare_kernel<64, true>, grid, 256, 0, stream, 1, pre);
    return int(e == cudaSuccess ? KVP_OK : KVP_ERR_CUDA);
  };
  const bool direct = n_jt == 1 && !dq_last;   // bwd_kernel writes dQ
  const bool read_first = f32 != nullptr && f32->read_first;
  for (int l0 = 0; read_first && l0 < s->L; l0 += MAX_GROUP) {   // the pre-passes of all layers, which clear nothing
    const int n = std::min(MAX_GROUP, s->L - l0);
    AuxParams ax = {};
    for (int i = 0; i < n; ++i) {
      ax.d_o[i] = reinterpret_cast<const __nv_bfloat16*>(d_o[l0 + i]);
      ax.delta[i] = reinterpret_cast<float*>(wsb + size_t(l0 + i) * delta_bytes);
    }
    ax.B = s->B;
    ax.S = s->S;
    ax.Hq = s->Hq;
    const int rc = prepare_f32(ax, n, reinterpret_cast<const float* const*>(o) + l0, f32->d_o + l0);
    if (rc != KVP_OK) return rc;
  }
  while (gi < groups.size()) {
    BwdParams p;
    const float *o32[MAX_GROUP] = {}, *do32[MAX_GROUP] = {};
    AuxParams ax = {};
    int slots = 0, ng = 0;
    p.cta_begin[0] = 0;
    p.first_slot[0] = 0;
    while (gi < groups.size() && slots + groups[gi].n <= MAX_GROUP) {
      const Group& g = groups[gi];
      int rc = make_map_bshd(&p.map_k[ng], k[g.owner], s->B, s->S, s->Hkv, dh, BT);
      if (rc == KVP_OK) rc = make_map_bshd(&p.map_v[ng], v[g.owner], s->B, s->S, s->Hkv, dh, BT);
      if (rc != KVP_OK) return rc;
      for (int i = 0; i < g.n; ++i) {
        const int l = g.members[i];
        rc = make_map_bshd(&p.map_q[slots], q[l], s->B, s->S, s->Hq, dh, BQ2);
        if (rc == KVP_OK) rc = make_map_bshd(&p.map_do[slots], d_o[l], s->B, s->S, s->Hq, dh, BQ2);
        if (rc != KVP_OK) return rc;
        p.lse[slots] = lse[l];
        p.delta[slots] = ax.delta[slots] = reinterpret_cast<float*>(wsb + size_t(l) * delta_bytes);
        p.dq_acc[slots] = reinterpret_cast<float*>(acc_base + size_t(slots) * acc_bytes);
        ax.d_o[slots] = reinterpret_cast<const __nv_bfloat16*>(d_o[l]);
        if (f32 != nullptr) {
          o32[slots] = reinterpret_cast<const float*>(o[l]);
          do32[slots] = f32->d_o[l];
        } else {
          ax.o[slots] = reinterpret_cast<const __nv_bfloat16*>(o[l]);
        }
        p.dq[slots] = ax.dq[slots] = dq[l];
        ax.dq_acc[slots] = p.dq_acc[slots];
        ++slots;
      }
      ax.dk_sum[ng] = dk_sum[g.owner];
      ax.dv_sum[ng] = dv_sum[g.owner];
      rc = make_map_sum(&p.map_dk[ng], dk_sum[g.owner], s->B, s->S, s->Hkv, dh);
      if (rc == KVP_OK) rc = make_map_sum(&p.map_dv[ng], dv_sum[g.owner], s->B, s->S, s->Hkv, dh);
      if (rc != KVP_OK) return rc;
      const BwdCut cut = bwd_cut(sizes, g.n * G, target);
      p.window[ng] = cut.window;
      p.parts[ng] = cut.parts;
      p.ctas_per_pair[ng] = 0;
      for (int w = 0; w * p.window[ng] < n_qt; ++w)
        p.ctas_per_pair[ng] += causal ? std::min(n_jt, ((w + 1) * p.window[ng] * BQ2 + BT - 1) / BT) : n_jt;
      p.ctas_per_pair[ng] *= p.parts[ng];
      p.first_slot[ng + 1] = slots;
      p.cta_begin[ng + 1] = p.cta_begin[ng] + n_pairs * p.ctas_per_pair[ng];
      ++ng;
      ++gi;
    }
    for (int i = slots; i < MAX_GROUP; ++i) {   // unused entries repeat slot 0, so that no descriptor is left unset
      p.map_q[i] = p.map_q[0];
      p.map_do[i] = p.map_do[0];
      p.lse[i] = p.lse[0];
      p.delta[i] = p.delta[0];
      p.dq_acc[i] = p.dq_acc[0];
      p.dq[i] = p.dq[0];
    }
    for (int i = ng; i < MAX_GROUP; ++i) {
      p.map_k[i] = p.map_k[0];
      p.map_v[i] = p.map_v[0];
      p.map_dk[i] = p.map_dk[0];
      p.map_dv[i] = p.map_dv[0];
      p.window[i] = p.window[0];
      p.parts[i] = p.parts[0];
      p.ctas_per_pair[i] = p.ctas_per_pair[0];
      p.first_slot[i + 1] = slots;
      p.cta_begin[i + 1] = p.cta_begin[ng];
    }
    p.n_classes = bwd_longest_first(sizes, slots, steps_per_sm, (long long)s->B * s->S * s->Hq, dh)
                      ? longest_first(p, ng, n_pairs, n_jt, n_qt, G, causal)
                      : 0;
    p.n_groups = ng;
    p.B = s->B;
    p.S = s->S;
    p.Hq = s->Hq;
    p.Hkv = s->Hkv;
    p.causal = causal;
    p.scale = sc;
    p.scale_log2 = sc * 1.4426950408889634f;
    ax.n_groups = ng;
    p.dq_f32 = ax.dq_f32 = f32 != nullptr;
    ax.B = s->B;
    ax.S = s->S;
    ax.Hq = s->Hq;
    p.dq_direct = direct;
    ax.acc_v4 = direct ? 0 : dq_acc_floats(s->B, s->S, s->Hq, dh) / 4;
    ax.kv_v4 = size_t(s->B) * s->S * s->Hkv * dh / 4;
    ax.scale = sc;
    timing_before(KVP_KERNEL_ATTN_BWD_AUX, stream);
    cudaError_t e = cudaSuccess;
    if (f32 != nullptr && !read_first) {
      const int rc = prepare_f32(ax, slots, o32, do32);
      if (rc != KVP_OK) return rc;
    } else {
      PrepareParams<false> pre;
      static_cast<AuxParams&>(pre) = ax;
      if (read_first) pre.B = 0;   // no rows: it only clears
      e = launch_kernel(dh == 128 ? bwd_prepare_kernel<128, false> : bwd_prepare_kernel<64, false>, aux_grid(8, slots), 256, 0, stream, 1, pre);
    }
    timing_after(KVP_KERNEL_ATTN_BWD_AUX, stream);
    if (e != cudaSuccess) return KVP_ERR_CUDA;
    dim3 grid(p.cta_begin[ng]);
    timing_before(KVP_KERNEL_ATTN_BWD, stream);
    e = dh == 128 ? launch_kernel(bwd_kernel<128>, grid, BWD_THREADS, BwdSmem<128>::TOTAL, stream, 1, p)
                  : launch_kernel(bwd_kernel<64>, grid, BWD_THREADS, BwdSmem<64>::TOTAL, stream, 1, p);
    timing_after(KVP_KERNEL_ATTN_BWD, stream);
    if (e != cudaSuccess) return KVP_ERR_CUDA;
    if (direct) continue;
    timing_before(KVP_KERNEL_ATTN_BWD_AUX, stream);
    e = launch_kernel(dh == 128 ? dq_convert_kernel<128> : dq_convert_kernel<64>, aux_grid(16, slots), 256, 0, stream, 1, ax);
    timing_after(KVP_KERNEL_ATTN_BWD_AUX, stream);
    if (e != cudaSuccess) return KVP_ERR_CUDA;
  }
  return KVP_OK;
}

}  // namespace kvp
