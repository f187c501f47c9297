// bf16 GEMM on tcgen05 tensor cores with TMEM accumulators, operands staged by TMA.
// Used for the Q / K / V / output projections (Eq. 1 of the paper) and their chain rule.  Four kernels; gemm_kernel:
//
// One persistent CTA per SM walks 128 x 256 output tiles.  Warp 0 issues TMA loads into a
// 4-stage shared-memory ring, warp 1 issues tcgen05.mma into one of two 256-column TMEM
// accumulators, warps 2-5 drain the other accumulator (tcgen05.ld -> registers -> shared memory ->
// TMA stores), so the epilogue of tile i overlaps the main loop of tile i+1.  Either operand may be K-major or
// MN-major in memory; that only changes the TMA box and the shared-memory descriptor.
// The K extent may be split over up to three operand pairs ("segments") that accumulate into the
// same tile, which is how dX = dQ Wq + dK Wk + dV Wv is produced with one output pass.
// One launch walks the tiles of a whole list of problems (different shapes, operands, operand modes and output
// types): the Q, K and V projections of every layer are one launch, so are all weight and input gradients of a
// backward pass, and the SMs idle only behind the last tile of the list instead of behind each GEMM's last wave.
#include <algorithm>
#include <type_traits>

#include "kvp_gemm_choice.h"
#include "kvp_host.h"
#include "kvp_sm100.cuh"

namespace kvp {
namespace {

constexpr int BM = GEMM_BM, BN = 256, BK = GEMM_BK, STAGES = 4;
constexpr int A_BYTES = BM * BK * 2;            // 16 KB
constexpr int B_BYTES = BN * BK * 2;            // 32 KB
constexpr int STAGE_BYTES = A_BYTES + B_BYTES;  // 48 KB
constexpr int GEMM_THREADS = 192;
constexpr int MAX_SEG = 3;
constexpr int GROUP_M = 16;  // m-tiles per rasterisation group (keeps an A slab resident in L2)
constexpr int EPI_BYTES = 4 * 2 * 4096;         // per epilogue warp two pieces of 32 rows x 128 bytes of C
constexpr size_t GEMM_SMEM = 1024 + size_t(STAGES) * STAGE_BYTES + EPI_BYTES + 256;
constexpr int MAX_PROB = 32;   // problems per launch
constexpr int MAX_MAPS = 96;   // tensor maps per launch (two per segment)

__device__ int g_gemm_status;

struct Problem {
  int M, N;
  int m_tiles, n_tiles;
  int tile_end;            // one past this problem's last tile in the launch's tile order
  int nseg;
  int kblocks[MAX_SEG];    // k-blocks (of BK) per segment
  int total_kb;
  short map_a[MAX_SEG];    // indices into GemmParams::maps
  short map_b[MAX_SEG];
  int a_mn, b_mn;
  int out_f32;
  uint32_t idesc;
};

struct GemmParams {
  CUtensorMap maps[MAX_MAPS];
  CUtensorMap map_c[MAX_PROB];   // C, box of 32 rows x 128 bytes
  Problem prob[MAX_PROB];
  int nprob;
  int total_tiles;
  // Self-test of the bounded waits (0 in every ordinary launch): the k-block count, plus one, at which the MMA
  // warp of CTA 0 withholds the arrival that frees a ring stage, and the wait limit that launch runs with.
  int withhold_at;
  unsigned long long wait_limit_ns;
};

// Position of tile t inside its problem: groups of GROUP_M m-tiles are walked n-tile by n-tile, which keeps an
// A slab resident in L2 while the B tiles stream past it.
__device__ __forceinline__ void tile_coords(int within_problem, int m_tiles, int n_tiles, int& tm, int& tn) {
  const int per_group = GROUP_M * n_tiles;
  const int g = within_problem / per_group;
  const int within = within_problem - g * per_group;
  const int gm = min(GROUP_M, m_tiles - g * GROUP_M);
  tm = g * GROUP_M + within % gm;
  tn = within / gm;
}

// One warp's 32 rows of a tile of C, from row0 and column n0 on: accumulator -> registers -> shared memory (128-byte
// swizzle) -> TMA stores of 32 rows x 128 bytes, two of them in flight; `release` when the accumulator has been read.  Stored
// from registers instead, a lane a row and 16 bytes at a time (half-sectors of 32 lines an instruction), a launch's last tile
// took 4 us after its last MMA (128 x 256, bf16), and a prompt of 347 tokens through a stage, nine launches of 129 to 144
// tiles among its 51, 811 us; 796 so.
template <typename F>
__device__ __forceinline__ void store_rows(const CUtensorMap* map, uint32_t taddr, int row0, int M, int n0, int N, int out_f32,
                                           uint8_t* stage, uint32_t& pieces, F release) {
  const int lane = lane_id();
  const int step = out_f32 ? 32 : 64;   // columns of 128 bytes
  const int end = row0 < M ? min(BN, N - n0) : 0;
  if (end <= 0) release();
#pragma unroll 1
  for (int c0 = 0; c0 < end; c0 += step, ++pieces) {
    uint8_t* const piece = stage + (pieces & 1) * 4096;
    uint32_t v[32];
    if (out_f32) {
      tmem_ld_x32(taddr + c0, v);
      tmem_ld_wait();
      if (out_f32 == OUT_F32_OF_BF16)
#pragma unroll
        for (int i = 0; i < 32; ++i) v[i] = bf16_bits_f32(__uint_as_float(v[i]));
    } else {
      uint32_t r[64];
      tmem_ld_x32(taddr + c0, *reinterpret_cast<uint32_t(*)[32]>(&r[0]));
      tmem_ld_x32(taddr + c0 + 32, *reinterpret_cast<uint32_t(*)[32]>(&r[32]));
      tmem_ld_wait();
#pragma unroll
      for (int i = 0; i < 32; ++i) v[i] = pack_bf16(__uint_as_float(r[2 * i]), __uint_as_float(r[2 * i + 1]));
    }
    if (c0 + step >= end) release();
    if (lane == 0) asm volatile("cp.async.bulk.wait_group.read 1;" ::: "memory");   // the piece before the last has been read
    __syncwarp();
#pragma unroll
    for (int j = 0; j < 8; ++j)
      *reinterpret_cast<uint4*>(piece + sw128_offset(lane, j)) = make_uint4(v[4 * j], v[4 * j + 1], v[4 * j + 2], v[4 * j + 3]);
    fence_proxy_async_smem();
    __syncwarp();
    if (lane == 0) {
      tma_store_2d(map, piece, n0 + c0, row0);
      asm volatile("cp.async.bulk.commit_group;" ::: "memory");
    }
  }
}

__global__ void __launch_bounds__(GEMM_THREADS, 1) gemm_kernel(const __grid_constant__ GemmParams p) {
  extern __shared__ uint8_t smem_raw[];
  uint8_t* smem = reinterpret_cast<uint8_t*>((reinterpret_cast<uintptr_t>(smem_raw) + 1023) & ~uintptr_t(1023));
  uint8_t* epi = smem + size_t(STAGES) * STAGE_BYTES;
  uint64_t* bars = reinterpret_cast<uint64_t*>(epi + EPI_BYTES);
  uint64_t* full = bars;                  // [STAGES]
  uint64_t* empty = bars + STAGES;        // [STAGES]
  uint64_t* acc_full = bars + 2 * STAGES; // [2]
  uint64_t* acc_empty = acc_full + 2;     // [2]
  uint32_t* tmem_slot = reinterpret_cast<uint32_t*>(acc_empty + 2);

  const int warp = threadIdx.x >> 5;
  const int lane = threadIdx.x & 31;
  int* err = &g_gemm_status;
  const int total_tiles = p.total_tiles;

  if (threadIdx.x == 0) {
    for (int s = 0; s < STAGES; ++s) {
      mbar_init(&full[s], 1);
      mbar_init(&empty[s], 1);
    }
    for (int a = 0; a < 2; ++a) {
      mbar_init(&acc_full[a], 1);
      mbar_init(&acc_empty[a], 4);
    }
    mbar_fence_init();
  }
  if (warp == 1) {
    tmem_alloc(tmem_slot, 512);
    tmem_relinquish();
  }
  tc_fence_before_sync();
  __syncthreads();
  tc_fence_after_sync();
  const uint32_t tmem_base = *tmem_slot;
  grid_dep_wait();

  if (warp == 0) {
    // ------------------------------ TMA producer ------------------------------
    {
      const uint32_t leader = elect_one();  // the whole warp runs the loop; one lane issues
      uint32_t it = 0;
      bool ok = true;
      int pi = 0;
      for (int t = blockIdx.x; t < total_tiles && ok; t += gridDim.x) {
        while (t >= p.prob[pi].tile_end) ++pi;
        const Problem& pr = p.prob[pi];
        int tm, tn;
        tile_coords(t - (pi ? p.prob[pi - 1].tile_end : 0), pr.m_tiles, pr.n_tiles, tm, tn);
        const int m0 = tm * BM, n0 = tn * BN;
        const int a_mn = pr.a_mn, b_mn = pr.b_mn;
        for (int seg = 0; seg < pr.nseg && ok; ++seg) {
          const CUtensorMap* map_a = &p.maps[pr.map_a[seg]];
          const CUtensorMap* map_b = &p.maps[pr.map_b[seg]];
          const int nkb = pr.kblocks[seg];
          for (int kb = 0; kb < nkb; ++kb, ++it) {
            const int s = it % STAGES;
            const uint32_t ph = (it / STAGES) & 1;
            if (!mbar_wait(&empty[s], ph ^ 1, err, p.wait_limit_ns)) { ok = false; break; }
            uint8_t* sa = smem + size_t(s) * STAGE_BYTES;
            uint8_t* sb = sa + A_BYTES;
            mbar_expect_tx_e(&full[s], STAGE_BYTES, leader);
            const int k0 = kb * BK;
            if (a_mn == 0) {
              tma_load_2d_e(sa, map_a, &full[s], k0, m0, leader);
            } else {
#pragma unroll
              for (int j = 0; j < BM / 64; ++j) tma_load_2d_e(sa + j * 8192, map_a, &full[s], m0 + 64 * j, k0, leader);
            }
            if (b_mn == 0) {
              tma_load_2d_e(sb, map_b, &full[s], k0, n0, leader);
            } else {
#pragma unroll
              for (int j = 0; j < BN / 64; ++j) tma_load_2d_e(sb + j * 8192, map_b, &full[s], n0 + 64 * j, k0, leader);
            }
          }
        }
      }
      grid_dep_launch();   // all loads are out: the next kernel may come up while the last tiles are finished
    }
  } else if (warp == 1) {
    // ------------------------------ MMA issuer ------------------------------
    {
      const uint32_t leader = elect_one();  // the whole warp runs the loop; one lane issues
      uint32_t it = 0;
      uint32_t tile_i = 0;
      bool ok = true;
      int pi = 0;
      for (int t = blockIdx.x; t < total_tiles && ok; t += gridDim.x, ++tile_i) {
        while (t >= p.prob[pi].tile_end) ++pi;
        const Problem& pr = p.prob[pi];
        const uint32_t a_step = pr.a_mn ? 2048u : 32u;   // bytes per 16-deep K step
        const uint32_t b_step = pr.b_mn ? 2048u : 32u;
        const uint32_t a_lbo = pr.a_mn ? 8192u : 0u;
        const uint32_t b_lbo = pr.b_mn ? 8192u : 0u;
        const uint32_t idesc = pr.idesc;
        const int total_kb = pr.total_kb;
        const int acc = tile_i & 1;
        const uint32_t acc_ph = (tile_i >> 1) & 1;
        if (!mbar_wait(&acc_empty[acc], acc_ph ^ 1, err, p.wait_limit_ns)) { ok = false; break; }
        tc_fence_after_sync();
        const uint32_t d_tmem = tmem_base + acc * BN;
        for (int kb = 0; kb < total_kb; ++kb, ++it) {
          const int s = it % STAGES;
          const uint32_t ph = (it / STAGES) & 1;
          if (!mbar_wait(&full[s], ph, err, p.wait_limit_ns)) { ok = false; break; }
          tc_fence_after_sync();
          const uint32_t sa = smem_u32(smem + size_t(s) * STAGE_BYTES);
          const uint32_t sb = sa + A_BYTES;
#pragma unroll
          for (int k = 0; k < BK / 16; ++k) {
            const uint64_t da = smem_desc_sw128(sa + k * a_step, a_lbo, 1024);
            const uint64_t db = smem_desc_sw128(sb + k * b_step, b_lbo, 1024);
            umma_ss(d_tmem, da, db, idesc, (kb | k) != 0, leader);
          }
          // frees the smem stage once these MMAs have read it
          if (!(p.withhold_at != 0 && blockIdx.x == 0 && it + 1 == uint32_t(p.withhold_at))) umma_commit(&empty[s], leader);
        }
        if (ok) umma_commit(&acc_full[acc], leader);
      }
    }
  } else {
    // ------------------------------ epilogue (warps 2..5) ------------------------------
    const int quarter = warp & 3;  // TMEM lane quarter this warp may access
    uint32_t tile_i = 0, pieces = 0;
    int pi = 0;
    for (int t = blockIdx.x; t < total_tiles; t += gridDim.x, ++tile_i) {
      while (t >= p.prob[pi].tile_end) ++pi;
      const Problem& pr = p.prob[pi];
      int tm, tn;
      tile_coords(t - (pi ? p.prob[pi - 1].tile_end : 0), pr.m_tiles, pr.n_tiles, tm, tn);
      const int acc = tile_i & 1;
      const uint32_t acc_ph = (tile_i >> 1) & 1;
      bool ok = mbar_wait(&acc_full[acc], acc_ph, err, p.wait_limit_ns);
      if (!__all_sync(0xffffffffu, ok)) break;
      tc_fence_after_sync();
      store_rows(&p.map_c[pi], tmem_base + (uint32_t(quarter * 32) << 16) + acc * BN, tm * BM + quarter * 32, pr.M, tn * BN, pr.N,
                 pr.out_f32, epi + quarter * 8192, pieces, [&]() {
                   tc_fence_before_sync();
                   __syncwarp();
                   if (lane == 0) mbar_arrive(&acc_empty[acc]);
                 });
    }
    if (lane == 0) asm volatile("cp.async.bulk.wait_group.read 0;" ::: "memory");   // before the shared memory goes away
    __syncwarp();
  }

  // ------------------------------ teardown ------------------------------
  tc_fence_before_sync();
  __syncthreads();
  if (warp == 1) {
    tc_fence_after_sync();
    tmem_dealloc(tmem_base, 512);
  }
}


// ------------------------------------------------------------------------------------------------------------
// The same GEMM on CTA pairs: 256 x 256 output tiles, one per pair of SMs (a cluster of two CTAs).  Each CTA of the
// pair loads 128 rows of A and 128 of the tile's 256 rows of B per k-block (32 KB per stage instead of 48 KB, so
// the ring is six stages deep) and drains its own 128 accumulator rows; the even CTA issues the M = 256 MMAs for
// both.  An MMA then reads 8 KB of operands per SM where the single-CTA tile reads 12 KB, which takes the shared-
// memory port off the critical path.  Barriers: full[s] lives in the even CTA and counts the bytes of both CTAs'
// loads; empty[s] and acc_full[a] exist in both CTAs and receive one MMA-completion arrival each; acc_empty[a]
// lives in the even CTA and collects the eight epilogue warps of the pair.
// ------------------------------------------------------------------------------------------------------------
constexpr int PBM = GEMM_PAIR_BM;                 // tile rows per pair
constexpr int PHALF = 128;                        // rows of A, and rows of B, per CTA
constexpr int PSTAGES = 6;
constexpr int PA_BYTES = PHALF * BK * 2;          // 16 KB
constexpr int PB_BYTES = PHALF * BK * 2;          // 16 KB
constexpr int PSTAGE_BYTES = PA_BYTES + PB_BYTES; // 32 KB per CTA
constexpr size_t PAIR_SMEM = 1024 + size_t(PSTAGES) * PSTAGE_BYTES + EPI_BYTES + 256;

__global__ void __cluster_dims__(2, 1, 1) __launch_bounds__(GEMM_THREADS, 1)
    gemm_pair_kernel(const __grid_constant__ GemmParams p) {
  extern __shared__ uint8_t smem_raw[];
  uint8_t* smem = reinterpret_cast<uint8_t*>((reinterpret_cast<uintptr_t>(smem_raw) + 1023) & ~uintptr_t(1023));
  uint8_t* epi = smem + size_t(PSTAGES) * PSTAGE_BYTES;
  uint64_t* bars = reinterpret_cast<uint64_t*>(epi + EPI_BYTES);
  uint64_t* full = bars;                    // [PSTAGES]  (used in the even CTA)
  uint64_t* empty = bars + PSTAGES;         // [PSTAGES]
  uint64_t* acc_full = bars + 2 * PSTAGES;  // [2]
  uint64_t* acc_empty = acc_full + 2;       // [2]        (used in the even CTA)
  uint32_t* tmem_slot = reinterpret_cast<uint32_t*>(acc_empty + 2);

  const int warp = threadIdx.x >> 5;
  const int lane = threadIdx.x & 31;
  int* err = &g_gemm_status;
  const int total_tiles = p.total_tiles;
  const uint32_t rank = cluster_ctarank();  // 0: issues the MMAs; 1: partner
  const int pair = blockIdx.x >> 1;
  const int n_pairs = gridDim.x >> 1;

  if (threadIdx.x == 0) {
    for (int s = 0; s < PSTAGES; ++s) {
      mbar_init(&full[s], 1);
      mbar_init(&empty[s], 1);
    }
    for (int a = 0; a < 2; ++a) {
      mbar_init(&acc_full[a], 1);
      mbar_init(&acc_empty[a], 8);
    }
    mbar_fence_init();
  }
  if (warp == 1) {
    tmem_alloc_pair(tmem_slot, 512);
    tmem_relinquish_pair();
  }
  tc_fence_before_sync();
  __syncthreads();
  cluster_sync_all();  // the partner's barriers exist before anything of this CTA can signal them
  tc_fence_after_sync();
  const uint32_t tmem_base = *tmem_slot;
  grid_dep_wait();

  if (warp == 0) {
    // ------------------------------ TMA producer (both CTAs) ------------------------------
    {
      const uint32_t leader = elect_one();
      uint32_t it = 0;
      bool ok = true;
      int pi = 0;
      for (int t = pair; t < total_tiles && ok; t += n_pairs) {
        while (t >= p.prob[pi].tile_end) ++pi;
        const Problem& pr = p.prob[pi];
        int tm, tn;
        tile_coords(t - (pi ? p.prob[pi - 1].tile_end : 0), pr.m_tiles, pr.n_tiles, tm, tn);
        const int m0 = tm * PBM + int(rank) * PHALF, n0 = tn * BN + int(rank) * PHALF;
        const int a_mn = pr.a_mn, b_mn = pr.b_mn;
        for (int seg = 0; seg < pr.nseg && ok; ++seg) {
          const CUtensorMap* map_a = &p.maps[pr.map_a[seg]];
          const CUtensorMap* map_b = &p.maps[pr.map_b[seg]];
          const int nkb = pr.kblocks[seg];
          for (int kb = 0; kb < nkb; ++kb, ++it) {
            const int s = it % PSTAGES;
            const uint32_t ph = (it / PSTAGES) & 1;
            if (!mbar_wait(&empty[s], ph ^ 1, err, p.wait_limit_ns)) { ok = false; break; }
            uint8_t* sa = smem + size_t(s) * PSTAGE_BYTES;
            uint8_t* sb = sa + PA_BYTES;
            if (rank == 0) mbar_expect_tx_e(&full[s], 2 * PSTAGE_BYTES, leader);   // both CTAs' bytes
            const uint32_t bar = cluster_addr_of(&full[s], 0);
            const int k0 = kb * BK;
            if (a_mn == 0) {
              tma_load_2d_pair_e(sa, map_a, bar, k0, m0, leader);
            } else {
#pragma unroll
              for (int j = 0; j < PHALF / 64; ++j) tma_load_2d_pair_e(sa + j * 8192, map_a, bar, m0 + 64 * j, k0, leader);
            }
            if (b_mn == 0) {
              tma_load_2d_pair_e(sb, map_b, bar, k0, n0, leader);
            } else {
#pragma unroll
              for (int j = 0; j < PHALF / 64; ++j) tma_load_2d_pair_e(sb + j * 8192, map_b, bar, n0 + 64 * j, k0, leader);
            }
          }
        }
      }
      grid_dep_launch();   // all loads are out: the next kernel may come up while the last tiles are finished
    }
  } else if (warp == 1) {
    // ------------------------------ MMA issuer (even CTA only) ------------------------------
    if (rank == 0) {
      const uint32_t leader = elect_one();
      uint32_t it = 0;
      uint32_t tile_i = 0;
      bool ok = true;
      int pi = 0;
      for (int t = pair; t < total_tiles && ok; t += n_pairs, ++tile_i) {
        while (t >= p.prob[pi].tile_end) ++pi;
        const Problem& pr = p.prob[pi];
        const uint32_t a_step = pr.a_mn ? 2048u : 32u;   // bytes per 16-deep K step
        const uint32_t b_step = pr.b_mn ? 2048u : 32u;
        const uint32_t a_lbo = pr.a_mn ? 8192u : 0u;
        const uint32_t b_lbo = pr.b_mn ? 8192u : 0u;
        const uint32_t idesc = pr.idesc;
        const int total_kb = pr.total_kb;
        const int acc = tile_i & 1;
        const uint32_t acc_ph = (tile_i >> 1) & 1;
        if (!mbar_wait(&acc_empty[acc], acc_ph ^ 1, err, p.wait_limit_ns)) { ok = false; break; }
        tc_fence_after_sync();
        const uint32_t d_tmem = tmem_base + acc * BN;
        for (int kb = 0; kb < total_kb; ++kb, ++it) {
          const int s = it % PSTAGES;
          const uint32_t ph = (it / PSTAGES) & 1;
          if (!mbar_wait(&full[s], ph, err, p.wait_limit_ns)) { ok = false; break; }
          tc_fence_after_sync();
          const uint32_t sa = smem_u32(smem + size_t(s) * PSTAGE_BYTES);
          const uint32_t sb = sa + PA_BYTES;
#pragma unroll
          for (int k = 0; k < BK / 16; ++k) {
            const uint64_t da = smem_desc_sw128(sa + k * a_step, a_lbo, 1024);
            const uint64_t db = smem_desc_sw128(sb + k * b_step, b_lbo, 1024);
            umma_ss_pair(d_tmem, da, db, idesc, (kb | k) != 0, leader);
          }
          // frees the stage in both CTAs once these MMAs have read it
          if (!(p.withhold_at != 0 && pair == 0 && it + 1 == uint32_t(p.withhold_at))) {
            umma_commit_pair(cluster_addr_of(&empty[s], 0), leader);
            umma_commit_pair(cluster_addr_of(&empty[s], 1), leader);
          }
        }
        if (ok) {
          umma_commit_pair(cluster_addr_of(&acc_full[acc], 0), leader);
          umma_commit_pair(cluster_addr_of(&acc_full[acc], 1), leader);
        }
      }
    }
  } else {
    // ------------------------------ epilogue (warps 2..5 of both CTAs) ------------------------------
    const int quarter = warp & 3;  // TMEM lane quarter this warp may access
    uint32_t tile_i = 0, pieces = 0;
    int pi = 0;
    for (int t = pair; t < total_tiles; t += n_pairs, ++tile_i) {
      while (t >= p.prob[pi].tile_end) ++pi;
      const Problem& pr = p.prob[pi];
      int tm, tn;
      tile_coords(t - (pi ? p.prob[pi - 1].tile_end : 0), pr.m_tiles, pr.n_tiles, tm, tn);
      const int acc = tile_i & 1;
      const uint32_t acc_ph = (tile_i >> 1) & 1;
      bool ok = mbar_wait(&acc_full[acc], acc_ph, err, p.wait_limit_ns);
      if (!__all_sync(0xffffffffu, ok)) break;
      tc_fence_after_sync();
      store_rows(&p.map_c[pi], tmem_base + (uint32_t(quarter * 32) << 16) + acc * BN, tm * PBM + int(rank) * PHALF + quarter * 32,
                 pr.M, tn * BN, pr.N, pr.out_f32, epi + quarter * 8192, pieces, [&]() {
                   tc_fence_before_sync();
                   __syncwarp();
                   if (lane == 0) mbar_arrive_cluster(cluster_addr_of(&acc_empty[acc], 0));
                 });
    }
    if (lane == 0) asm volatile("cp.async.bulk.wait_group.read 0;" ::: "memory");   // before the shared memory goes away
    __syncwarp();
  }

  // ------------------------------ teardown ------------------------------
  // Neither CTA may leave, or free its TMEM, while the partner can still signal its barriers or while MMAs of the
  // pair can still write its accumulator: both wait for each other first.
  tc_fence_before_sync();
  __syncthreads();
  cluster_sync_all();
  if (warp == 1) {
    tc_fence_after_sync();
    tmem_dealloc_pair(tmem_base, 512);
  }
}

// ------------------------------------------------------------------------------------------------------------
// Few rows of A (the tokens of a decode step): C^T = B A^T, K split over a cluster.
//
// With at most 128 rows of A the product is bound by reading B once, and the 128 x 256 tiles above put it on N / 256
// CTAs: 16 of 148 SMs at N = 4096, 29 us for 33.5 MB.  Here B supplies the M = 128 side of the MMA and the tokens its
// N side (a multiple of 16, so 16 tokens cost 16 columns and not 128 rows), and the k-blocks of a tile are dealt to
// the CTAs of a cluster, each with its own ring and one or two accumulators.  The partials meet in shared memory: every CTA
// moves its accumulators from TMEM to shared memory as [token][128 columns] fp32 and sums its share of the tokens over the
// cluster's accumulators through distributed shared memory, in their order along K, so results depend neither on timing nor on
// how many accumulators a CTA has.
// Measured (us, K x N at M tokens; 128 x 256 tiles -> this kernel; reading B at the copy rate): 4096 x 4096 at 16
// tokens 28.7 -> 11.6 (5.2), 4096 x 11008 at 16 30.8 -> 20.6 (13.9), 11008 x 4096 at 16 65.5 -> 20.6 (13.9), 4096 x
// 4096 at 128 28.9 -> 14.5 (5.5); a launch that does almost nothing takes 6.
// In clusters of one and two, where a warp has more than two tokens to sum, it takes four at a time with two partials: one
// token and partial after the other, each waiting for the other CTA's shared memory, took 4.5 of the 16 us of 347 x 4096 x 4096
// (back to back 21.2 -> 16.8; 347 x 4096 x 11008 40.8 -> 32.8).  In larger clusters a warp has fewer tokens, and the longer code
// takes more to fetch than it saves: 129 x 4096 x 4096, four CTAs, 13.7 -> 14.5, 128 x 1024 x 1024, eight, 8.0 -> 9.3.
// ------------------------------------------------------------------------------------------------------------
constexpr int SROWS = SPLIT_COLS;                // rows of B (output columns) per tile: the M of the MMA
constexpr int SB_BYTES = SPLIT_B_BYTES;          // 16 KB
constexpr int SPLIT_THREADS = 192;
// k-blocks of B a CTA asks into L2 before the kernels ahead of it have finished (a token step's 56 kernels: 601 us
// without, 595 with 8, 613 with 32)
constexpr int SPLIT_PREFETCH = 8;

struct SplitProblem {
  int M, N;
  int tok_tiles;           // token tiles of `nt` rows
  int tile_end;
  int kblocks;
  int out_f32;
  long long ldc;
  void* c;
};
template <int NP>
struct SplitParams {
  CUtensorMap map_a[NP], map_b[NP];
  SplitProblem prob[NP];
  int nt;                  // tokens per tile: the N of the MMA, a multiple of 16
  int stages;
  int tmem_cols;
  uint32_t idesc;
};

// WIDE: four tokens a warp at a time.  PARTS: accumulators of a CTA (one or two), each with a run of its k-blocks.  STREAM: B,
// which one CTA reads once, is marked first to go in L2 (stream_weights, kvp_gemm_choice.h).
template <int NP, bool WIDE, int PARTS, bool STREAM>
__global__ void __launch_bounds__(SPLIT_THREADS, 4) gemm_split_kernel(const __grid_constant__ SplitParams<NP> p) {
  extern __shared__ uint8_t smem_raw[];
  uint8_t* smem = reinterpret_cast<uint8_t*>((reinterpret_cast<uintptr_t>(smem_raw) + 1023) & ~uintptr_t(1023));
  __shared__ uint64_t full[SPLIT_MAX_STAGES], empty[SPLIT_MAX_STAGES], acc_full;
  __shared__ uint32_t tmem_slot;

  const int warp = threadIdx.x >> 5;
  const int lane = threadIdx.x & 31;
  int* err = &g_gemm_status;
  const uint32_t split = cluster_nctarank(), rank = cluster_ctarank();
  const int t = blockIdx.x / split;
  const int stages = p.stages, nt = p.nt;
  const int stage_bytes = SB_BYTES + nt * (BK * 2);

  int pi = 0;
  if constexpr (NP > 1)
    while (t >= p.prob[pi].tile_end) ++pi;
  const SplitProblem& pr = p.prob[pi];
  const int within = t - (pi ? p.prob[pi - 1].tile_end : 0);
  const int n0 = (within / pr.tok_tiles) * SROWS;   // first output column (row of B)
  const int m0 = (within % pr.tok_tiles) * nt;      // first token
  const int pieces = int(split) * PARTS, piece = int(rank) * PARTS;   // of K, and this CTA's first
  const int kb0 = piece * pr.kblocks / pieces, kb1 = (piece + PARTS) * pr.kblocks / pieces;

  if (threadIdx.x == 0) {
    for (int s = 0; s < stages; ++s) {
      mbar_init(&full[s], 1);
      mbar_init(&empty[s], 1);
    }
    mbar_init(&acc_full, 1);
    mbar_fence_init();
  }
  if (warp == 1) {
    tmem_alloc(&tmem_slot, p.tmem_cols);
    tmem_relinquish();
  }
  tc_fence_before_sync();
  __syncthreads();
  tc_fence_after_sync();
  const uint32_t tmem_base = tmem_slot;
  grid_dep_launch();
  // while the kernels ahead of this one finish, the first k-blocks of B come into L2 (a prefetch reads nothing yet)
  if (warp == 0) {
    const uint32_t leader = elect_one();
    for (int kb = kb0; kb < min(kb1, kb0 + SPLIT_PREFETCH); ++kb) tma_prefetch_2d_e(&p.map_b[pi], kb * BK, n0, leader);
  }
  grid_dep_wait();

  if (warp == 0) {
    const uint32_t leader = elect_one();
    const uint64_t policy = STREAM ? l2_evict_first() : 0;
    int s = 0;
    uint32_t ph = 1;
    for (int kb = kb0; kb < kb1; ++kb) {
      if (!mbar_wait(&empty[s], ph, err)) break;
      uint8_t* sb = smem + s * stage_bytes;
      mbar_expect_tx_e(&full[s], stage_bytes, leader);
      if constexpr (STREAM) tma_load_2d_e(sb, &p.map_b[pi], &full[s], kb * BK, n0, policy, leader);
      else tma_load_2d_e(sb, &p.map_b[pi], &full[s], kb * BK, n0, leader);
      tma_load_2d_e(sb + SB_BYTES, &p.map_a[pi], &full[s], kb * BK, m0, leader);
      if (++s == stages) {
        s = 0;
        ph ^= 1;
      }
    }
  } else if (warp == 1) {
    const uint32_t leader = elect_one();
    int s = 0;
    uint32_t ph = 0;
    bool ok = true;
    const int kb_second = PARTS == 2 ? (piece + 1) * pr.kblocks / pieces : kb1;
    for (int kb = kb0; kb < kb1; ++kb) {
      if (!mbar_wait(&full[s], ph, err)) { ok = false; break; }
      tc_fence_after_sync();
      const uint32_t acc = kb < kb_second ? tmem_base : tmem_base + p.tmem_cols / 2;
      const uint32_t b_lo = desc_lo_sw128(smem_u32(smem + s * stage_bytes), 0);
      const uint32_t a_lo = desc_lo_sw128(smem_u32(smem + s * stage_bytes + SB_BYTES), 0);
#pragma unroll
      for (int k = 0; k < BK / 16; ++k)
        umma_ss_w(acc, desc_lo_add(b_lo, k * 32), desc_lo_add(a_lo, k * 32), desc_hi_sw128(1024), p.idesc,
                  (kb != kb0 && (PARTS == 1 || kb != kb_second)) || k != 0, leader);
      umma_commit(&empty[s], leader);
      if (++s == stages) {
        s = 0;
        ph ^= 1;
      }
    }
    if (ok) umma_commit(&acc_full, leader);
  }
  // every warp waits for the accumulators; the four warps that own their lanes move them to shared memory as [token][128]
  // fp32 (the ring is idle now), one behind the other
  __syncwarp();
  float* part = reinterpret_cast<float*>(smem);
  bool ok = mbar_wait(&acc_full, 0, err);
  ok = __all_sync(0xffffffffu, ok);
  if (ok && warp >= 2) {
    tc_fence_after_sync();
    const int quarter = warp & 3;
    uint32_t taddr = tmem_base + (uint32_t(quarter * 32) << 16);
    float* dst = part + quarter * 32 + lane;
#pragma unroll 1
    for (int i = 0; i < PARTS; ++i, taddr += p.tmem_cols / 2, dst += nt * SROWS) {
      int c0 = 0;
      if constexpr (WIDE) {
        for (; c0 + 32 <= nt; c0 += 32) {
          uint32_t r[32];
          tmem_ld_x32(taddr + c0, r);
          tmem_ld_wait();
#pragma unroll
          for (int k = 0; k < 32; ++k) dst[(c0 + k) * SROWS] = __uint_as_float(r[k]);
        }
      }
      for (; c0 < nt; c0 += 16) {
        uint32_t r[16];
        tmem_ld_x16(taddr + c0, r);
        tmem_ld_wait();
#pragma unroll
        for (int k = 0; k < 16; ++k) dst[(c0 + k) * SROWS] = __uint_as_float(r[k]);
      }
    }
    tc_fence_before_sync();
  }
  __syncthreads();
  if (split > 1) cluster_sync_all();
  // each CTA of the cluster sums its share of the tokens over all partials, always in their order along K
  if (ok) {
    const int col = n0 + lane * 4;
    const uint32_t mine = smem_u32(part) + lane * 16;
    const int n_tok = min(nt, pr.M - m0);
    const int step = int(split) * (SPLIT_THREADS / 32);
    auto store = [&](int tk, float4 acc) {
      if (col >= pr.N) return;
      const size_t at = size_t(m0 + tk) * pr.ldc + col;
      if (pr.out_f32) {
        if (pr.out_f32 == OUT_F32_OF_BF16)
          acc = make_float4(__uint_as_float(bf16_bits_f32(acc.x)), __uint_as_float(bf16_bits_f32(acc.y)),
                            __uint_as_float(bf16_bits_f32(acc.z)), __uint_as_float(bf16_bits_f32(acc.w)));
        *reinterpret_cast<float4*>(reinterpret_cast<float*>(pr.c) + at) = acc;
      } else
        *reinterpret_cast<uint2*>(reinterpret_cast<__nv_bfloat16*>(pr.c) + at) =
            make_uint2(pack_bf16(acc.x, acc.y), pack_bf16(acc.z, acc.w));
    };
    // a warp's tokens U at a time, and J partials: the loads of other CTAs' shared memory overlap
    constexpr int U = WIDE ? 4 : 1, J = WIDE ? 2 : 4;
    for (int tk = int(rank) + warp * int(split); tk < n_tok; tk += step * U) {
      float4 acc[U];
#pragma unroll
      for (int u = 0; u < U; ++u) acc[u] = make_float4(0.f, 0.f, 0.f, 0.f);
#pragma unroll 1
      for (int j0 = 0; j0 < pieces; j0 += J) {
        float4 v[J][U];
#pragma unroll
        for (int j = 0; j < J; ++j) {
          const int from = min(j0 + j, pieces - 1);
          const uint32_t peer = cluster_map_addr(mine + from % PARTS * (nt * SROWS * 4), from / PARTS);
#pragma unroll
          for (int u = 0; u < U; ++u)
            if (tk + u * step < n_tok && j0 + j < pieces) v[j][u] = ld_cluster_f4(peer + (tk + u * step) * (SROWS * 4));
        }
#pragma unroll
        for (int j = 0; j < J; ++j)
#pragma unroll
          for (int u = 0; u < U; ++u)
            if (tk + u * step < n_tok && j0 + j < pieces) {
              acc[u].x += v[j][u].x;
              acc[u].y += v[j][u].y;
              acc[u].z += v[j][u].z;
              acc[u].w += v[j][u].w;
            }
      }
#pragma unroll
      for (int u = 0; u < U; ++u)
        if (tk + u * step < n_tok) store(tk + u * step, acc[u]);
    }
  }
  __syncthreads();
  if (split > 1) cluster_sync_all();   // no CTA leaves while a peer may still read its partial
  if (warp == 1) {
    tc_fence_after_sync();
    tmem_dealloc(tmem_base, p.tmem_cols);
  }
}

// ------------------------------------------------------------------------------------------------------------
// Up to a few thousand rows of A (prompts, small batches), and the gradients: CTA pairs with the operands swapped,
// C^T = B A^T.
//
// Each pair of CTAs owns 256 columns of C (rows of B: 128 a CTA, the M = 256 of the pair's MMA) and a tile of tokens (the
// N, split between the CTAs' loads).  256 x 256 tiles of gemm_pair_kernel pad 347 tokens to 512; here the tokens are cut
// into tiles of up to 256, in steps of 32.  Forward they are all of one size, walked column by column, so that the columns'
// weights come from memory once.  Gradients have whole tiles and one of the remainder (in steps of 128 where A is MN-major:
// its TMA boxes hold 64 rows and each CTA loads half of the tile), dealt out by cost (kvp_gemm_choice.h).  A lane of the
// epilogue holds a column, so a warp stores rows of 64
// consecutive bytes, two at a time (128 in fp32), where a lane of gemm_pair_kernel's holds a row.  Roles, segments and
// barriers are those of gemm_pair_kernel, the ring has as many stages as tiles of the launch's size leave room for;
// results are bit-identical to its (same products, same order along K).
// Bound: the 120 GB/s that an SM draws from L2 (tiles of up to 192 tokens), then the tensor pipe.  Measured (us, weights
// not in L2; gemm_pair_kernel -> this, tokens x columns x K): 347 x 32000 x 4096 102 -> 82, 512 x 11008 x 4096 51 -> 40, 1500 x
// 4096 x 11008 155 -> 121, 2328 x 4096 x 4096 90 -> 70.  A ring of 7 to 9 stages instead of 6 gave 2 to 8 %.  With a
// short K the stores bound it, and four epilogue warps leave them waiting for one another: sixteen instead of four took
// fp32 results of 2328 x 1024 x 1024, four problems, from 48 to 24 us and those of 776 tokens, six problems, from 26 to
// 16 (bf16: 13.8 -> 14.6; the same change slowed gemm_kernel and gemm_pair_kernel by 2 to 10 %).
// ------------------------------------------------------------------------------------------------------------
constexpr int TCOLS = 256;                        // columns of C per pair
constexpr int TMAX_STAGES = 10;                   // a stage holds, per CTA, 128 rows of B and half of a tile's rows of A
// Four for every quarter of the TMEM lanes, taking 32 tokens each in turn: all on every tile, or (gradient launches in which pairs
// have several tiles of few k-blocks) eight on every other one, so that the stores of one tile run while the other eight wait for the
// next and read it out.  With all sixteen on each the stores of a tile of fp32 results went out at 6.7 TB/s, and nothing for as
// long again.  Measured (us, sixteen -> eight): 264 tokens, 7 layers of d 1024 74 -> 69; 128 tokens, 8 layers of d 4096 232 -> 216; but
// 2328 tokens, 3 layers of d 1024 36 -> 39, where the last tiles count.  Forward, with K up to 768, it makes no
// difference (four of 2048 x 4096 x 512 44.6 -> 44.8, three of 3000 x 4096 x 768 70.6 -> 69.0, runs 2 apart) or one either way (fp32
// results, eight layers of d 512, 700 tokens 78.3 -> 76.8, of d 256, 500 tokens, heads of 64 28.5 -> 30.3).
constexpr int TALL_EPI_WARPS = 16, TALL_ALTERNATE_ROUNDS = 6, TALL_SHORT_KBLOCKS = 12;
constexpr int TALL_THREADS = (2 + TALL_EPI_WARPS) * 32;
constexpr int TALL_RING = 224 * 1024;             // the ring takes as many stages as fit
constexpr int TALL_SMEM = 1024 + TALL_RING + 256;

struct TallList {                                 // the tiles of one problem that have the same number of tokens
  int prob;
  int nt;                                         // tokens (rows of C) per tile, a multiple of 32; of 128 if A is MN-major
  int m_first, n_tok;                             // first token, tiles along the tokens
  float inv_n_tok;
  int tile_end;                                   // one past the list's last tile in the launch's tile order
  uint32_t idesc;
  short map_a[MAX_SEG];                           // per segment; the box holds half of a tile's tokens
};
struct TallProblem {
  int M, N, nseg, kblocks[MAX_SEG], total_kb;
  short map_b[MAX_SEG];
  int a_mn, b_mn, out_f32;
  long long ldc;
  void* c;
};
template <bool DEAL>
struct TallDeal {                                 // gradients: the pairs' tiles, class by class (0 classes: pairs take tiles in turn)
  int n_classes;
  uint16_t first[DEAL_CLASSES][DEAL_PAIRS + 1];
};
template <>
struct TallDeal<false> {
  static constexpr int n_classes = 0;
};
template <int NP, int NSEG, bool DEAL>            // problems, and segments of all of them, that the parameter block holds
struct TallParams {
  TallDeal<DEAL> deal;
  CUtensorMap map_b[NSEG], map_a[2 * NSEG];
  TallProblem prob[NP];
  TallList list[2 * NP];
  int total_tiles;
  int stages, stage_bytes;
  int alternate;                                  // eight epilogue warps a tile
};

template <int NP, int NSEG, bool DEAL>
__global__ void __cluster_dims__(2, 1, 1) __launch_bounds__(TALL_THREADS, 1)
    gemm_tall_kernel(const __grid_constant__ TallParams<NP, NSEG, DEAL> p) {
  extern __shared__ uint8_t smem_raw[];
  uint8_t* smem = reinterpret_cast<uint8_t*>((reinterpret_cast<uintptr_t>(smem_raw) + 1023) & ~uintptr_t(1023));
  uint64_t* bars = reinterpret_cast<uint64_t*>(smem + TALL_RING);
  uint64_t* full = bars;                        // [stages]  (used in the even CTA)
  uint64_t* empty = bars + TMAX_STAGES;         // [stages]
  uint64_t* acc_full = bars + 2 * TMAX_STAGES;  // [2]
  uint64_t* acc_empty = acc_full + 2;       // [2]        (used in the even CTA)
  uint32_t* tmem_slot = reinterpret_cast<uint32_t*>(acc_empty + 2);

  const int warp = threadIdx.x >> 5;
  const int lane = threadIdx.x & 31;
  int* err = &g_gemm_status;
  const int total_tiles = p.total_tiles, stages = p.stages, stage_bytes = p.stage_bytes;
  const uint32_t rank = cluster_ctarank();  // 0: issues the MMAs; 1: partner
  const int pair = blockIdx.x >> 1;
  const int n_pairs = gridDim.x >> 1;

  if (threadIdx.x == 0) {
    for (int s = 0; s < stages; ++s) {
      mbar_init(&full[s], 1);
      mbar_init(&empty[s], 1);
    }
    for (int a = 0; a < 2; ++a) {
      mbar_init(&acc_full[a], 1);
      mbar_init(&acc_empty[a], 2 * TALL_EPI_WARPS >> p.alternate);
    }
    mbar_fence_init();
  }
  if (warp == 1) {
    tmem_alloc_pair(tmem_slot, 512);
    tmem_relinquish_pair();
  }
  tc_fence_before_sync();
  __syncthreads();
  cluster_sync_all();  // the partner's barriers exist before anything of this CTA can signal them
  tc_fence_after_sync();
  const uint32_t tmem_base = *tmem_slot;
  grid_dep_wait();

  struct Tile {
    int li, prob, nt, m0, n0;
    int turn, t;   // next tile: round (tiles in turn) or class, and its number there
  };
  // The pair's next tile; li only grows.  In turn: rounds of n_pairs tiles, dealt forwards and backwards.
  auto next_tile = [&](Tile& w) -> bool {
    int t;
    bool dealt = false;
    if constexpr (DEAL) {
      dealt = p.deal.n_classes > 0;
      if (dealt) {
        while (w.t >= p.deal.first[w.turn][pair + 1]) {
          if (++w.turn == p.deal.n_classes) return false;
          w.t = p.deal.first[w.turn][pair];
        }
        t = w.t++;
      }
    }
    if (!dealt) {
      do {
        if (w.turn * n_pairs >= total_tiles) return false;
        t = w.turn * n_pairs + ((w.turn & 1) ? n_pairs - 1 - pair : pair);
        ++w.turn;
      } while (t >= total_tiles);   // only the last round can be short
    }
    while (t >= p.list[w.li].tile_end) ++w.li;
    const TallList& l = p.list[w.li];
    const int within = t - (w.li ? p.list[w.li - 1].tile_end : 0);
    w.prob = l.prob;
    w.nt = l.nt;
    int column = int(float(within) * l.inv_n_tok), tok = within - column * l.n_tok;   // (right to within one, for up to 2^24 tiles)
    if (tok < 0) {
      --column;
      tok += l.n_tok;
    } else if (tok >= l.n_tok) {
      ++column;
      tok -= l.n_tok;
    }
    w.m0 = l.m_first + tok * l.nt;
    w.n0 = column * TCOLS;
    return true;
  };
  auto first_tile = [&]() {
    Tile w{};
    if constexpr (DEAL)
      if (p.deal.n_classes > 0) w.t = p.deal.first[0][pair];
    return w;
  };

  if (warp == 0) {
    // ------------------------------ TMA producer (both CTAs) ------------------------------
    const uint32_t leader = elect_one();
    int s = 0;
    uint32_t ph = 1;
    bool ok = true;
    Tile w = first_tile();
    while (ok && next_tile(w)) {
      const TallProblem& pr = p.prob[w.prob];
      const int half = w.nt / 2, a_mn = pr.a_mn, b_mn = pr.b_mn;
      const uint32_t bytes = 2u * uint32_t(PA_BYTES + half * (BK * 2));   // of both CTAs
      const int n0 = w.n0 + int(rank) * 128, m0 = w.m0 + int(rank) * half;
      for (int seg = 0; seg < pr.nseg && ok; ++seg) {
        const CUtensorMap* map_b = &p.map_b[pr.map_b[seg]];
        const CUtensorMap* map_a = &p.map_a[p.list[w.li].map_a[seg]];
        const int nkb = pr.kblocks[seg];
        for (int kb = 0; kb < nkb; ++kb) {
          if (!mbar_wait(&empty[s], ph, err)) { ok = false; break; }
          uint8_t* sb = smem + s * stage_bytes;
          uint8_t* sa = sb + PA_BYTES;
          if (rank == 0) mbar_expect_tx_e(&full[s], bytes, leader);
          const uint32_t bar = cluster_addr_of(&full[s], 0);
          if (b_mn == 0) {
            tma_load_2d_pair_e(sb, map_b, bar, kb * BK, n0, leader);
          } else {
#pragma unroll
            for (int j = 0; j < 2; ++j) tma_load_2d_pair_e(sb + j * 8192, map_b, bar, n0 + 64 * j, kb * BK, leader);
          }
          if (a_mn == 0) {
            tma_load_2d_pair_e(sa, map_a, bar, kb * BK, m0, leader);
          } else {
            for (int j = 0; j < half / 64; ++j) tma_load_2d_pair_e(sa + j * 8192, map_a, bar, m0 + 64 * j, kb * BK, leader);
          }
          if (++s == stages) {
            s = 0;
            ph ^= 1;
          }
        }
      }
    }
    grid_dep_launch();   // all loads are out: the next kernel may come up while the last tiles are finished
  } else if (warp == 1) {
    // ------------------------------ MMA issuer (even CTA only) ------------------------------
    if (rank == 0) {
      const uint32_t leader = elect_one();
      int s = 0;
      uint32_t ph = 0, tile_i = 0;
      bool ok = true;
      Tile w = first_tile();
      while (ok && next_tile(w)) {
        const uint32_t idesc = p.list[w.li].idesc;
        const TallProblem& pr = p.prob[w.prob];
        const int nkb = pr.total_kb;
        const uint32_t a_step = pr.a_mn ? 2048u : 32u, b_step = pr.b_mn ? 2048u : 32u;   // bytes per 16-deep K step
        const uint32_t a_lbo = pr.a_mn ? 8192u : 0u, b_lbo = pr.b_mn ? 8192u : 0u;
        const int acc = tile_i & 1;
        if (!mbar_wait(&acc_empty[acc], ((tile_i >> 1) & 1) ^ 1, err)) { ok = false; break; }
        tc_fence_after_sync();
        const uint32_t d_tmem = tmem_base + acc * 256;
        for (int kb = 0; kb < nkb; ++kb) {
          if (!mbar_wait(&full[s], ph, err)) { ok = false; break; }
          tc_fence_after_sync();
          const uint32_t sb = smem_u32(smem + s * stage_bytes);
#pragma unroll
          for (int k = 0; k < BK / 16; ++k)
            umma_ss_pair(d_tmem, smem_desc_sw128(sb + k * b_step, b_lbo, 1024), smem_desc_sw128(sb + PA_BYTES + k * a_step, a_lbo, 1024),
                         idesc, (kb | k) != 0, leader);
          umma_commit_pair(cluster_addr_of(&empty[s], 0), leader);
          umma_commit_pair(cluster_addr_of(&empty[s], 1), leader);
          if (++s == stages) {
            s = 0;
            ph ^= 1;
          }
        }
        if (ok) {
          umma_commit_pair(cluster_addr_of(&acc_full[acc], 0), leader);
          umma_commit_pair(cluster_addr_of(&acc_full[acc], 1), leader);
        }
        ++tile_i;
      }
    }
  } else {
    // ------------------------------ epilogue (warps 2.. of both CTAs): lane = column of C ------------------------------
    const int quarter = warp & 3;  // TMEM lane quarter this warp may access
    const bool alternate = p.alternate;
    const int group = alternate ? (warp - 2) >> 3 : 0, step = alternate ? 64 : 128;
    const int first = 32 * ((warp - 2) >> 2) & (step - 1);
    uint32_t tile_i = 0;
    Tile w = first_tile();
    for (; next_tile(w); ++tile_i) {
      const int acc = tile_i & 1;
      if (alternate && acc != group) continue;
      const TallProblem& pr = p.prob[w.prob];
      const bool ok = mbar_wait(&acc_full[acc], (tile_i >> 1) & 1, err);
      if (!__all_sync(0xffffffffu, ok)) break;
      tc_fence_after_sync();
      const int col = w.n0 + int(rank) * 128 + quarter * 32 + lane;
      const int n_tok = min(w.nt, pr.M - w.m0);
      const uint32_t taddr = tmem_base + (uint32_t(quarter * 32) << 16) + acc * 256;
      // 32 tokens at a time.  The accumulator is given back ahead of the last stores, by an arrival that does not wait for any.
#pragma unroll 1
      for (int c0 = first;; c0 += step) {
        uint32_t r[32];
        const bool last = c0 + step >= n_tok;
        if (c0 < n_tok) tmem_ld_x32(taddr + c0, r);
        tmem_ld_wait();
        if (last) {
          tc_fence_before_sync();
          __syncwarp();
          if (lane == 0) mbar_arrive_cluster_relaxed(cluster_addr_of(&acc_empty[acc], 0));
        }
        const int left = col < pr.N ? n_tok - c0 : 0;
        if (pr.out_f32) {
          if (pr.out_f32 == OUT_F32_OF_BF16)
#pragma unroll
            for (int i = 0; i < 32; ++i) r[i] = bf16_bits_f32(__uint_as_float(r[i]));
          float* dst = reinterpret_cast<float*>(pr.c) + size_t(w.m0 + c0) * pr.ldc + col;
#pragma unroll
          for (int i = 0; i < 32; ++i, dst += pr.ldc)
            if (i < left) *dst = __uint_as_float(r[i]);
        } else if (c0 < n_tok) {
          // two tokens at a time: even lanes end up with two columns of the first, odd lanes with two of the second
          const int odd = lane & 1;
          __nv_bfloat16* dst = reinterpret_cast<__nv_bfloat16*>(pr.c) + size_t(w.m0 + c0 + odd) * pr.ldc + (col - odd);
#pragma unroll
          for (int i = 0; i < 32; i += 2, dst += 2 * pr.ldc) {
            const uint32_t got = __shfl_xor_sync(0xffffffffu, odd ? r[i] : r[i + 1], 1);
            const float lo = __uint_as_float(odd ? got : r[i]), hi = __uint_as_float(odd ? r[i + 1] : got);
            if (i + odd < left) *reinterpret_cast<uint32_t*>(dst) = pack_bf16(lo, hi);
          }
        }
        if (last) break;
      }
    }
  }

  // ------------------------------ teardown: as gemm_pair_kernel ------------------------------
  tc_fence_before_sync();
  __syncthreads();
  cluster_sync_all();
  if (warp == 1) {
    tc_fence_after_sync();
    tmem_dealloc_pair(tmem_base, 512);
  }
}

}  // namespace

int gemm_read_status() {
  int v = 0;
  if (cudaMemcpyFromSymbol(&v, g_gemm_status, sizeof(int)) != cudaSuccess) return -1;
  if (v != 0) {
    int zero = 0;
    cudaMemcpyToSymbol(g_gemm_status, &zero, sizeof(int));
  }
  return v;
}

namespace {

int check_problem(const GemmProblem& g) {
  if (g.M <= 0 || g.N <= 0 || g.nseg < 1 || g.nseg > MAX_SEG || g.c == nullptr) return KVP_ERR_INVALID_ARG;
  if ((g.N % 8) != 0 || (g.ldc % 8) != 0 || !aligned16(g.c)) return KVP_ERR_UNSUPPORTED;
  for (int s = 0; s < g.nseg; ++s) {
    const GemmSeg& e = g.segs[s];
    if (e.a == nullptr || e.b == nullptr || e.K <= 0) return KVP_ERR_INVALID_ARG;
    if ((e.K % 8) != 0 || (e.lda % 8) != 0 || (e.ldb % 8) != 0 || !aligned16(e.a) || !aligned16(e.b))
      return KVP_ERR_UNSUPPORTED;
  }
  return KVP_OK;
}

// Tensor map of one operand with `rows` rows (of A) or columns (of B): K-major boxes hold box_rows of them by BK, MN-major
// ones 64 by BK.
int encode_operand(CUtensorMap* map, const void* base, int64_t ld, int rows, int K, int mn, uint32_t box_rows) {
  uint64_t dims[2] = {uint64_t(mn ? rows : K), uint64_t(mn ? K : rows)};
  uint64_t strides[1] = {uint64_t(ld) * 2};
  uint32_t box[2] = {mn ? 64u : uint32_t(BK), mn ? uint32_t(BK) : box_rows};
  return make_tensor_map(map, base, 2, 2, dims, strides, box, true);
}

int launch_group(const GemmProblem* probs, int n, cudaStream_t stream, int withhold_at, unsigned long long wait_limit_ns,
                 bool pair) {
  const int bm = pair ? PBM : BM;
  static thread_local GemmParams p;   // 19 KB: kept off the stack
  p.nprob = n;
  p.withhold_at = withhold_at;
  p.wait_limit_ns = wait_limit_ns != 0 ? wait_limit_ns : kWaitLimitNs;
  int n_maps = 0, tiles = 0;
  for (int i = 0; i < n; ++i) {
    const GemmProblem& g = probs[i];
    Problem& q = p.prob[i];
    q.M = g.M;
    q.N = g.N;
    q.m_tiles = (g.M + bm - 1) / bm;
    q.n_tiles = (g.N + BN - 1) / BN;
    tiles += q.m_tiles * q.n_tiles;
    q.tile_end = tiles;
    q.nseg = g.nseg;
    q.total_kb = 0;
    for (int s = 0; s < MAX_SEG; ++s) {
      q.kblocks[s] = 0;
      q.map_a[s] = q.map_b[s] = 0;
    }
    for (int s = 0; s < g.nseg; ++s) {
      q.kblocks[s] = (g.segs[s].K + BK - 1) / BK;
      q.total_kb += q.kblocks[s];
      q.map_a[s] = short(n_maps);
      q.map_b[s] = short(n_maps + 1);
      const GemmSeg& e = g.segs[s];
      int rc = encode_operand(&p.maps[n_maps], e.a, e.lda, g.M, e.K, g.a_mn, BM);
      if (rc == KVP_OK) rc = encode_operand(&p.maps[n_maps + 1], e.b, e.ldb, g.N, e.K, g.b_mn, pair ? PHALF : BN);
      if (rc != KVP_OK) return rc;
      n_maps += 2;
    }
    q.a_mn = g.a_mn;
    q.b_mn = g.b_mn;
    q.out_f32 = g.out_f32;
    q.idesc = umma_idesc_bf16(bm, BN, g.a_mn, g.b_mn);
    const int elem = g.out_f32 ? 4 : 2;
    const uint64_t dims[2] = {uint64_t(g.N), uint64_t(g.M)};
    const uint64_t strides[1] = {uint64_t(g.M > 1 ? g.ldc : (g.N + 7) / 8 * 8) * elem};
    const uint32_t box[2] = {uint32_t(128 / elem), 32};
    const int rc = make_tensor_map(&p.map_c[i], g.c, elem, 2, dims, strides, box, true);
    if (rc != KVP_OK) return rc;
  }
  for (int i = n; i < MAX_PROB; ++i) p.prob[i] = p.prob[n - 1];
  p.total_tiles = tiles;
  if ((pair ? allow_smem<gemm_pair_kernel>(int(PAIR_SMEM)) : allow_smem<gemm_kernel>(int(GEMM_SMEM))) != cudaSuccess) return KVP_ERR_CUDA;
  timing_before(KVP_KERNEL_GEMM, stream);
  const cudaError_t e =
      pair ? launch_kernel(gemm_pair_kernel, 2 * min(tiles, sm_count() / 2), GEMM_THREADS, PAIR_SMEM, stream, 1, p)
           : launch_kernel(gemm_kernel, min(tiles, sm_count()), GEMM_THREADS, GEMM_SMEM, stream, 1, p);
  timing_after(KVP_KERNEL_GEMM, stream);
  return e == cudaSuccess ? KVP_OK : KVP_ERR_CUDA;
}

constexpr int SPLIT_MAX_PROB = MAX_PROB;

// Both operands K-major, one segment: the shape of every forward projection.
bool k_major(const GemmProblem* probs, int n) {
  for (int i = 0; i < n; ++i)
    if (probs[i].nseg != 1 || probs[i].a_mn != 0 || probs[i].b_mn != 0) return false;
  return n > 0;
}

template <int NP, bool WIDE, int PARTS>
auto split_kernel(bool stream_b) -> decltype(&gemm_split_kernel<NP, WIDE, PARTS, true>) {
  if (stream_b) return allow_smem<gemm_split_kernel<NP, WIDE, PARTS, true>>(226 * 1024) == cudaSuccess ? &gemm_split_kernel<NP, WIDE, PARTS, true> : nullptr;
  return allow_smem<gemm_split_kernel<NP, WIDE, PARTS, false>>(226 * 1024) == cudaSuccess ? &gemm_split_kernel<NP, WIDE, PARTS, false> : nullptr;
}

template <int NP>
int launch_split(const GemmProblem* probs, int n, const SplitConfig& cfg, bool stream_b, cudaStream_t stream) {
  SplitParams<NP> p;
  int tiles = 0;
  for (int i = 0; i < n; ++i) {
    const GemmProblem& g = probs[i];
    SplitProblem& q = p.prob[i];
    q.M = g.M;
    q.N = g.N;
    q.tok_tiles = (g.M + cfg.nt - 1) / cfg.nt;
    tiles += q.tok_tiles * ((g.N + SROWS - 1) / SROWS);
    q.tile_end = tiles;
    q.kblocks = (g.segs[0].K + BK - 1) / BK;
    q.out_f32 = g.out_f32;
    q.ldc = g.ldc;
    q.c = g.c;
    const GemmSeg& e = g.segs[0];
    int rc = encode_operand(&p.map_a[i], e.a, e.lda, g.M, e.K, 0, uint32_t(cfg.nt));
    if (rc == KVP_OK) rc = encode_operand(&p.map_b[i], e.b, e.ldb, g.N, e.K, 0, SROWS);
    if (rc != KVP_OK) return rc;
  }
  p.nt = cfg.nt;
  p.stages = cfg.stages;
  p.tmem_cols = 32 * cfg.parts;
  while (p.tmem_cols < cfg.nt * cfg.parts) p.tmem_cols *= 2;
  p.idesc = umma_idesc_bf16(SROWS, cfg.nt, 0, 0);
  // Tensor memory is shared out in proportion to shared memory, so that CTAs of this kernel that fit on an SM by the latter
  // never wait for the former: a CTA that waits holds up the peers of its cluster.  40 KB keep it off the SMs of the GEMM
  // kernels that take all 512 columns, which have peers too, and of the attention backward and the forward at head size 128.
  // The forward at head size 64 (114 KB) can share an SM with it, and one of the two then waits in its allocation until the
  // other ends; it does end, for a CTA of the attention waits for no other CTA.
  const int ring = cfg.stages * (SB_BYTES + cfg.nt * BK * 2), part = cfg.parts * cfg.nt * SROWS * 4;
  const int smem = 1024 + std::max(std::max(ring, part), std::max(40 * 1024, p.tmem_cols * 440));
  const bool wide = cfg.split <= 2 && cfg.nt > 2 * cfg.split * (SPLIT_THREADS / 32);
  auto* const kernel = cfg.parts == 2 ? (wide ? split_kernel<NP, true, 2>(stream_b) : split_kernel<NP, false, 2>(stream_b))
                                      : (wide ? split_kernel<NP, true, 1>(stream_b) : split_kernel<NP, false, 1>(stream_b));
  if (kernel == nullptr) return KVP_ERR_CUDA;
  timing_before(KVP_KERNEL_GEMM, stream);
  const cudaError_t e = launch_kernel(kernel, tiles * cfg.split, SPLIT_THREADS, smem, stream, cfg.split, p);
  timing_after(KVP_KERNEL_GEMM, stream);
  return e == cudaSuccess ? KVP_OK : KVP_ERR_CUDA;
}

template <int NP, int NSEG, bool DEAL>
int launch_tall(const GemmProblem* probs, int n, int nt, bool even, cudaStream_t stream) {
  TallParams<NP, NSEG, DEAL> p;
  int lists = 0, tiles = 0, maps_a = 0, maps_b = 0;
  for (int i = 0; i < n; ++i) {
    const GemmProblem& g = probs[i];
    TallProblem& q = p.prob[i];
    q.M = g.M;
    q.N = g.N;
    q.nseg = g.nseg;
    q.total_kb = 0;
    q.a_mn = g.a_mn;
    q.b_mn = g.b_mn;
    q.out_f32 = g.out_f32;
    q.ldc = g.ldc;
    q.c = g.c;
    for (int e = 0; e < g.nseg; ++e) {
      const GemmSeg& sg = g.segs[e];
      q.kblocks[e] = (sg.K + BK - 1) / BK;
      q.total_kb += q.kblocks[e];
      q.map_b[e] = short(maps_b);
      const int rc = encode_operand(&p.map_b[maps_b++], sg.b, sg.ldb, g.N, sg.K, g.b_mn, 128);
      if (rc != KVP_OK) return rc;
    }
  }
  // Lists: forward the tiles of each problem, all of one size.  Gradients: whole tiles and one of the remainder, input gradients
  // (K-major A) of up to two tiles in equal ones; the costliest lists first.
  struct Part {
    int prob, nt, m_first, n_tok;
    float us;
  } parts[2 * NP];
  int n_parts = 0;
  for (int i = 0; i < n; ++i) {
    const GemmProblem& g = probs[i];
    const int unit = g.a_mn ? 128 : TALL_UNIT, most = (g.M + nt - 1) / nt;
    const bool equal = even || (!g.a_mn && most == 2);   // (a few rows more than one tile: both tiles read all of B)
    const int size = even ? nt : equal ? ((g.M + most - 1) / most + unit - 1) / unit * unit : nt;
    const int whole = equal ? (g.M + size - 1) / size : g.M / size, rest = std::max(0, g.M - whole * size);
    auto add = [&](int t, int first, int cnt) {
      if (cnt > 0) parts[n_parts++] = Part{i, t, first, cnt, even ? 0.f : gradient_tile_us(p.prob[i].total_kb, t, g.out_f32 != 0)};
    };
    add(size, 0, whole);
    add((rest + unit - 1) / unit * unit, whole * size, rest > 0 ? 1 : 0);
  }
  if (!even) std::stable_sort(parts, parts + n_parts, [](const Part& a, const Part& b) { return a.us > b.us; });
  int classes = 0, in_class[DEAL_CLASSES], short_tiles = 0;
  float class_us[DEAL_CLASSES];
  for (int i = 0; i < n_parts; ++i) {
    const Part& q = parts[i];
    const GemmProblem& g = probs[q.prob];
    TallList l{};
    l.prob = q.prob;
    l.nt = q.nt;
    l.m_first = q.m_first;
    l.n_tok = q.n_tok;
    l.inv_n_tok = 1.f / q.n_tok;
    const int here = q.n_tok * ((g.N + TCOLS - 1) / TCOLS);
    tiles += here;
    l.tile_end = tiles;
    l.idesc = umma_idesc_bf16(256, l.nt, g.b_mn, g.a_mn);
    for (int e = 0; e < g.nseg; ++e) {
      l.map_a[e] = short(maps_a);
      const int rc = encode_operand(&p.map_a[maps_a++], g.segs[e].a, g.segs[e].lda, g.M, g.segs[e].K, g.a_mn, uint32_t(l.nt / 2));
      if (rc != KVP_OK) return rc;
    }
    p.list[lists++] = l;
    if (classes == 0 || (q.us < class_us[classes - 1] && classes < DEAL_CLASSES)) {
      class_us[classes] = q.us;
      in_class[classes++] = 0;
    }
    in_class[classes - 1] += here;
    if (p.prob[q.prob].total_kb <= TALL_SHORT_KBLOCKS) short_tiles += here;
  }
  const int pairs = std::min(tiles, sm_count() / 2);
  if constexpr (DEAL) {
    p.deal.n_classes = !even && classes > 1 && in_class[0] < pairs && pairs <= DEAL_PAIRS && tiles <= 0xffff ? classes : 0;
    if (p.deal.n_classes > 0) deal_tiles(class_us, in_class, classes, pairs, p.deal.first);
  }
  p.total_tiles = tiles;
  p.stage_bytes = PA_BYTES + nt / 2 * (BK * 2);
  p.stages = std::min(TMAX_STAGES, TALL_RING / p.stage_bytes);
  p.alternate = !even && short_tiles >= TALL_ALTERNATE_ROUNDS * pairs;
  if (allow_smem<gemm_tall_kernel<NP, NSEG, DEAL>>(TALL_SMEM) != cudaSuccess) return KVP_ERR_CUDA;
  timing_before(KVP_KERNEL_GEMM, stream);
  const cudaError_t e = launch_kernel(gemm_tall_kernel<NP, NSEG, DEAL>, 2 * pairs, TALL_THREADS, TALL_SMEM, stream, 1, p);
  timing_after(KVP_KERNEL_GEMM, stream);
  return e == cudaSuccess ? KVP_OK : KVP_ERR_CUDA;
}

// 0: single-CTA tiles only; 1: whichever kernel suits the sizes; 2: CTA pairs (gemm_pair_kernel) everywhere.
// In modes 1 and 2 pairs are never used for a group with a problem of at most 128 rows (half of every pair tile would be
// padding).
int g_pair_mode = 1;

bool use_pair(const GemmProblem* probs, int n) {
  if (g_pair_mode == 0) return false;
  for (int i = 0; i < n; ++i)
    if (probs[i].M <= BM) return false;
  return true;
}

}  // namespace

void gemm_set_pair_mode(int mode) { g_pair_mode = mode; }
int gemm_pair_mode() { return g_pair_mode; }

namespace {

// Parameter blocks of four sizes: each 8 KB of them take 0.6 us to launch.  f is given the size.
template <typename F>
int by_count(int n, F f) {
  if (n == 1) return f(std::integral_constant<int, 1>());
  if (n <= 4) return f(std::integral_constant<int, 4>());
  if (n <= 8) return f(std::integral_constant<int, 8>());
  return f(std::integral_constant<int, MAX_PROB>());
}

// The gradient GEMMs of a launch (pair mode 1) run on gemm_tall_kernel, in tiles of 256 rows; of 128 where those would
// leave half of the pairs idle.  Measured (us, all weight and input gradients of a backward pass: gemm_kernel / tiles of
// 128 / 256): 256 tokens x 256, four layers 14.4 / 7.0 / 9.0; 400 x 4096, two layers 32.1 / 28.9 / 23.2; 1984 x 1024, six
// layers 70.6 / 72.8 / 59.3; 1664 x 4096, five layers 140 / 147 / 120; 4096 x 4096, one layer 303 / 352 / 282.
// With the costliest tiles first, two equal tiles where 256 rows leave a few, and accumulators given back without waiting for
// stores (an arrival with release semantics at cluster scope waits until all the thread's stores have reached L2): 264 tokens, 7
// layers of d 1024 102 -> 69; 288, 8 of 2048 79 -> 65; 128, 8 of 4096 250 -> 216; 264 with output projection, 2 of 4096 200 -> 140.
// Launches of more than GRADIENT_MAX_FLOP (about 0.3 ms) stay on gemm_kernel, although by themselves they too are a little
// faster on pairs (4096 x 4096, four layers, 0.8 TFLOP: 1140 / - / 1030): they belong to steps of many milliseconds, which
// the board's power limit bounds, and there the rest of the step slows by more than the pairs gain (training step of eight
// layers, 2 x 8192 tokens: 46.2 -> 47.8 ms; of four layers with output projections, 8 x 4096: 39.9 -> 41.4 ms).
constexpr double GRADIENT_MAX_FLOP = 5e11;
int gemm_gradient(const GemmProblem* probs, int n, cudaStream_t stream) {
  int tiles = 0, segs = 0;
  double flop = 0;
  for (int i = 0; i < n; ++i) {
    const GemmProblem& g = probs[i];
    tiles += ((g.M + 255) / 256) * ((g.N + TCOLS - 1) / TCOLS);
    segs += g.nseg;
    for (int e = 0; e < g.nseg; ++e) flop += 2.0 * g.M * g.N * g.segs[e].K;
  }
  if (flop > GRADIENT_MAX_FLOP) return launch_group(probs, n, stream, 0, 0, false);
  const int nt = 4 * tiles <= sm_count() ? 128 : 256;
  if (segs == 1) return launch_tall<1, 1, false>(probs, n, nt, false, stream);
  if (segs <= 4) return launch_tall<4, 4, true>(probs, n, nt, false, stream);
  if (n <= 8 && segs <= 12) return launch_tall<8, 12, true>(probs, n, nt, false, stream);
  return launch_tall<MAX_PROB, MAX_MAPS / 2, true>(probs, n, nt, false, stream);
}

// A forward GEMM (K-major operands, one segment): -1 when the tile kernels take it
int gemm_forward(const GemmProblem* probs, int n, cudaStream_t stream) {
  int rows = 0;
  for (int i = 0; i < n; ++i) rows = std::max(rows, probs[i].M);
  GemmSize sizes[MAX_PROB];
  auto sizes_of = [&](const GemmProblem* g, int cnt) {
    for (int i = 0; i < cnt; ++i) sizes[i] = GemmSize{g[i].M, g[i].N, g[i].segs[0].K};
    return sizes;
  };
  if (rows <= SPLIT_MAX_ROWS) {
    for (int begin = 0; begin < n; begin += SPLIT_MAX_PROB) {
      const int cnt = std::min(SPLIT_MAX_PROB, n - begin);
      const GemmProblem* g = probs + begin;
      const SplitConfig cfg = split_config(sizes_of(g, cnt), cnt, sm_count());
      const bool stream_b = stream_weights(sizes, cnt, cfg.nt);
      const int rc = by_count(cnt, [&](auto np) { return launch_split<np>(g, cnt, cfg, stream_b, stream); });
      if (rc != KVP_OK) return rc;
    }
    return KVP_OK;
  }
  if (g_pair_mode != 1 || rows > CHOICE_MAX_ROWS) return -1;
  for (int begin = 0; begin < n; begin += MAX_PROB) {
    const int cnt = std::min(MAX_PROB, n - begin);
    const GemmProblem* g = probs + begin;
    const Choice c = choose_forward(sizes_of(g, cnt), cnt, sm_count());
    int rc;
    if (c.kind == Choice::kTall) {
      rc = by_count(cnt, [&](auto np) { return launch_tall<np, np, false>(g, cnt, c.nt, true, stream); });
    } else if (c.kind == Choice::kSplit) {
      const SplitConfig cfg{c.nt, c.split, 1, std::min(SPLIT_MAX_STAGES, 220 * 1024 / (SB_BYTES + c.nt * BK * 2))};
      rc = by_count(cnt, [&](auto np) { return launch_split<np>(g, cnt, cfg, false, stream); });
    } else {
      rc = launch_group(g, cnt, stream, 0, 0, c.kind == Choice::kPair);
    }
    if (rc != KVP_OK) return rc;
  }
  return KVP_OK;
}

}  // namespace

int gemm_grouped(const GemmProblem* probs, int n, cudaStream_t stream) {
  if (n < 0 || (n > 0 && probs == nullptr)) return KVP_ERR_INVALID_ARG;
  for (int i = 0; i < n; ++i) {
    const int rc = check_problem(probs[i]);
    if (rc != KVP_OK) return rc;
  }
  const bool forward = k_major(probs, n);
  if (forward) {
    const int rc = gemm_forward(probs, n, stream);
    if (rc >= 0) return rc;
  }
  // as many problems per launch as the parameter block holds
  int begin = 0;
  while (begin < n) {
    int end = begin, maps = 0;
    while (end < n && end - begin < MAX_PROB && maps + 2 * probs[end].nseg <= MAX_MAPS) maps += 2 * probs[end++].nseg;
    const int rc = !forward && g_pair_mode == 1
                       ? gemm_gradient(probs + begin, end - begin, stream)
                       : launch_group(probs + begin, end - begin, stream, 0, 0, use_pair(probs + begin, end - begin));
    if (rc != KVP_OK) return rc;
    begin = end;
  }
  return KVP_OK;
}

int gemm_bf16(int M, int N, const GemmSeg* segs, int nseg, int a_mn, int b_mn, void* c, int64_t ldc, int out_f32,
              cudaStream_t stream, int withhold_at, unsigned long long wait_limit_ns) {
  if (nseg < 1 || nseg > MAX_SEG || segs == nullptr) return KVP_ERR_INVALID_ARG;
  GemmProblem g{};
  g.M = M;
  g.N = N;
  g.nseg = nseg;
  for (int s = 0; s < nseg; ++s) g.segs[s] = segs[s];
  g.a_mn = a_mn;
  g.b_mn = b_mn;
  g.c = c;
  g.ldc = ldc;
  g.out_f32 = out_f32;
  if (withhold_at == 0) return gemm_grouped(&g, 1, stream);
  const int rc = check_problem(g);
  return rc == KVP_OK ? launch_group(&g, 1, stream, withhold_at, wait_limit_ns, use_pair(&g, 1)) : rc;
}

}  // namespace kvp
