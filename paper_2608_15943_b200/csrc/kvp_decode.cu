// Split-KV decode attention over the shared paged cache, and the cache append.
//
// A unit is (donor group, sequence, KV head): its K/V rows are streamed from HBM exactly once and applied to every
// query row that reads them: the Hq/Hkv query heads of the KV head's group for the donor layer AND for each consumer
// layer of the group (Eq. 3 of the paper: consumers reuse the donor's K/V), up to 16 rows, as the M dimension of
// mma.sync m16n8k16 (bf16 in, fp32 accumulate).  The kernel is bound by HBM bandwidth, so the design is about bytes in
// flight and about every warp having the same share of them:
//  - The rows of all units form one list of 16-token granules (8 KB at dh 128: 4 KB of K, 4 KB of V; both contiguous,
//    a page block of one KV head is), in order of (group, sequence, KV head, position).  The lengths are in device
//    memory, so every block sums them up itself and takes an equal share of the list, wherever its ends fall: no
//    part-filled last wave, whatever the batch and the lengths.  (kvp_deal.h has the rules; the list has empty places that
//    stand for the merge of each unit.)  Long lists are cut into more shares than blocks that
//    fit, so that the block scheduler evens out SMs that draw memory at different rates.
//  - Short units, none of them much longer than an equal share, are not cut but dealt out whole, since every piece costs a
//    block a merge of its warps (30 sequences of 500 tokens, 8 groups at dh 64: 46 us by units, 96 us when each was cut in
//    two).
//  - The four warps of a block take the granules of a share in turn, each with a ring of its own filled by 16-byte
//    cp.async copies that are fully coalesced and continue across the ends of units; two blocks per SM.  (A contiguous
//    share for every warp instead read memory 3 % slower.)  No transposes in HBM -- V fragments come from ldmatrix.trans
//    on the swizzled ring.
//  - A unit that lies inside one share is finished there.  The pieces of the others, (max, sum, output) triples, at most
//    two per share, are merged by a second small kernel that finds them by the same arithmetic.
// Measured with the merge (us), against a grid of (unit, 2048-token split) blocks with a merge of one thread per output
// element: 16 sequences of 4096 tokens 61 -> 50 (the copy rate takes 41), 8 of 8K-16K in two groups 141 -> 128 (113), one
// of 65536 74 -> 49 (41), 2 of 16K in eight groups 172 -> 170, 3 of 3000 in six groups at dh 64 26.8 -> 27.1, 4 of 128K
// at 32 KV heads 1192 -> 1177 (1313), 32 of 16K-32K in six groups 2767 -> 2687.
#include <math.h>

#include <algorithm>
#include <mutex>

#include "kvp_deal.h"
#include "kvp_host.h"
#include "kvp_sm100.cuh"

namespace kvp {
namespace {

constexpr int DEC_WARPS = 4;
constexpr int DEC_THREADS = DEC_WARPS * 32;
constexpr int GRAN = 16;           // tokens per ring stage
constexpr int DEC_STAGES = 3;      // granules per warp in the ring
template <int DH>
constexpr int DEC_CTAS_PER_SM = DH == 128 ? 2 : 4;   // as many as shared memory holds
// P is rounded to bf16 against a reference that rises with the largest score so far and, every REFERENCE_GRANULES granules of
// a warp, falls to that of the granule, or to REFERENCE_DROP (log2) below the largest so far: the probabilities that raise it
// are exact, so that the error of O does not grow with the length of a share.  (2-norm, of which 1.66e-3 is the rounding of O
// itself to bf16, 32 sequences of 16K to 32K tokens: 2.23e-3 with a reference that never falls, 2.15e-3 with pieces of 32
// granules a warp, 2.12e-3 so, 0.6 % slower.  Against the largest of each granule by itself: 1.94e-3, 1.2 % slower.)
constexpr int REFERENCE_GRANULES = 16;
constexpr float REFERENCE_DROP = 8.f;
constexpr int MAX_DEC_GROUPS = 64, FEW_DEC_GROUPS = 8;   // a launch of few groups has a parameter block of 1 KB, not 8: 0.6 us less to launch
constexpr int MAX_MEMBERS = 4;     // layers of a donor group served by one pass (rows = members * G <= 16)

__device__ int g_dec_status;

struct DecGroup {
  const __nv_bfloat16* k_cache;
  const __nv_bfloat16* v_cache;
  const void* q[MAX_MEMBERS];            // [B,Hq,dh], bf16 or (io_f32) fp32
  void* o[MAX_MEMBERS];                  // [B,Hq,dh], bf16 or (io_f32) fp32
  float* lse[MAX_MEMBERS];               // [B,Hq]
  int n_members;
  int pad;
};

struct DecSizes {
  const int32_t* block_table;  // [B, max_pages]
  const int32_t* lengths;      // [B]
  float* part_o;               // [pieces][rows][DH]
  float* part_ml;              // [pieces][rows][2]
  int rows;                    // query rows of the largest group
  int n_groups, B, Hq, Hkv, page_size, max_pages, n_pages;
  int fit;                     // blocks that fit on the device
  int max_shares;              // most shares of the list
  int by_units;                // the lists are short at any length: whole units are dealt out, no sums are formed
  int num_splits;              // > 0: the caller's split count instead; a block is one (unit, split)
  int io_f32;                  // queries are read and outputs written as fp32 (rounded to bf16 on load / widened on store)
  float scale_log2;
};
template <int NG>
struct DecParams : DecSizes {
  DecGroup grp[NG];
};

__device__ __forceinline__ int clamp_length(const DecSizes& p, int len) { return min(max(len, 1), p.max_pages * p.page_size); }
__device__ __forceinline__ int clamped_length(const DecSizes& p, int b) { return clamp_length(p, p.lengths[b]); }
__device__ __forceinline__ int granules_of(int len) { return (len + GRAN - 1) / GRAN; }

// Over the batch, formed by one warp: granules (of one KV head) of the sequences before b_before, of all, and of the longest.
// len0: the length (unclamped) of the lane's sequence among the first 32.
__device__ __forceinline__ void sum_granules(const DecSizes& p, int len0, int b_before, int& before, int& all, int& longest) {
  const int lane = threadIdx.x & 31;
  int sum = 0, most = 0, first = 0;
  for (int b = lane; b < p.B; b += 32) {
    const int n = granules_of(clamp_length(p, b < 32 ? len0 : p.lengths[b]));
    sum += n;
    most = max(most, n);
    first += b < b_before ? n : 0;
  }
  all = __reduce_add_sync(0xffffffffu, sum);
  longest = __reduce_max_sync(0xffffffffu, most);
  before = b_before > 0 ? __reduce_add_sync(0xffffffffu, first) : 0;
}
// The lengths of the first 32 sequences, one a lane, before the kernels ahead have finished (through L2: no line of them may
// stay in L1, later loads must see what those kernels write).  What was worked out from them holds if they are still the same
// behind the wait, and is worked out again if not: the lengths of a step are in place long before.  Batches of more than 32
// only look behind it.  (From the wait to a block's first data went 4.2 to 6 us, most of it this arithmetic out of a cold
// instruction cache.  Append, decode and merge, us: 8 sequences of 8K-16K in four layers 133.4 -> 130.0, 15 of 2K-4K in six
// 40.5 -> 37.0, 8 of 12K in five 67.3 -> 63.3, 28 of 1000 in three 30.4 -> 28.3.)
__device__ __forceinline__ int early_length(const DecSizes& p) {
  const int lane = threadIdx.x & 31;
  return lane < p.B ? __ldcg(p.lengths + lane) : 0;
}
// The first T mod n of n shares of a list of T granules hold one more than the others.
struct Dealt {
  uint32_t q, r;
  __device__ __forceinline__ Dealt(long long total, uint32_t n) : q(uint32_t(div_places(total, n))), r(uint32_t(total - (long long)q * n)) {}
  __device__ __forceinline__ long long begin(uint32_t i) const { return (long long)i * q + min(i, r); }
  __device__ __forceinline__ uint32_t size(uint32_t i) const { return q + (i < r ? 1u : 0u); }
  __device__ __forceinline__ int share_of(long long g) const {
    const long long longer = (long long)r * (q + 1);
    return g < longer ? int(div_places(g, q + 1)) : int(r + div_places(g - longer, q));
  }
};

// 16-byte asynchronous copy; with src_bytes == 0 nothing is read and the destination is filled with zeros
__device__ __forceinline__ void cp_async16(uint32_t dst, const void* src, uint32_t src_bytes) {
  asm volatile("cp.async.cg.shared.global [%0], [%1], 16, %2;" ::"r"(dst), "l"(src), "r"(src_bytes) : "memory");
}
__device__ __forceinline__ void cp_async_commit() { asm volatile("cp.async.commit_group;" ::: "memory"); }
template <int N>
__device__ __forceinline__ void cp_async_wait() {
  asm volatile("cp.async.wait_group %0;" ::"n"(N) : "memory");
}
__device__ __forceinline__ void mma_bf16(float (&c)[4], uint32_t a0, uint32_t a1, uint32_t a2, uint32_t a3, uint32_t b0,
                                         uint32_t b1) {
  asm volatile(
      "mma.sync.aligned.m16n8k16.row.col.f32.bf16.bf16.f32 {%0,%1,%2,%3}, {%4,%5,%6,%7}, {%8,%9}, {%0,%1,%2,%3};"
      : "+f"(c[0]), "+f"(c[1]), "+f"(c[2]), "+f"(c[3])
      : "r"(a0), "r"(a1), "r"(a2), "r"(a3), "r"(b0), "r"(b1));
}
__device__ __forceinline__ float fast_exp2(float x) {
  float y;
  asm("ex2.approx.ftz.f32 %0, %1;" : "=f"(y) : "f"(x));
  return y;
}

// ln(l 2^m), with the sum of the two logarithms and the constant kept to twice the precision before the only rounding
__device__ __forceinline__ float log_sum(float m, float l) {
  const float t = log2f(l), s = m + t, b = s - m;
  const float low = (m - (s - b)) + (t - b);          // s + low == m + t
  constexpr double kLn2 = 0.693147180559945309417;
  constexpr float hi = float(kLn2), lo = float(kLn2 - double(hi));
  return fmaf(s, hi, fmaf(s, lo, low * hi));
}

// Ring stage layout: GRAN rows of DH bf16 (DH*2 bytes per row) for K, then the same for V.  The
// 16-byte chunk index is XOR-ed with (row & 7) so that ldmatrix reads are bank-conflict free.
template <int DH>
__device__ __forceinline__ uint32_t ring_off(int row, int chunk) {
  return uint32_t(row) * (DH * 2) + (uint32_t(chunk ^ (row & 7)) << 4);
}

template <int DH, int NG>
__global__ void __launch_bounds__(DEC_THREADS, DEC_CTAS_PER_SM<DH>) decode_kernel(const __grid_constant__ DecParams<NG> p) {
  constexpr int ROW_BYTES = DH * 2;
  constexpr int CHUNKS = ROW_BYTES / 16;           // 16-byte chunks per row
  constexpr int TILE_BYTES = GRAN * ROW_BYTES;     // K (or V) part of a stage
  constexpr int STAGE_BYTES = 2 * TILE_BYTES;
  constexpr int STAGES = DEC_STAGES;
  constexpr int CP_PER_LANE = TILE_BYTES / 16 / 32;
  constexpr int KSTEPS = DH / 16;
  constexpr int NBLK = DH / 8;

  extern __shared__ __align__(128) uint8_t dsmem[];
  const int warp = threadIdx.x >> 5;
  const int lane = threadIdx.x & 31;
  const int g = lane >> 2, t = lane & 3;
  const int G = p.Hq / p.Hkv;
  __shared__ float2 s_o[DEC_WARPS - 1][NBLK * 32]; // eight rows of the results that warp 0 merges into its own
  __shared__ float2 s_ml[DEC_WARPS - 1][32];
  // A position in the list of granules: unit (grp, b, hk), granule `gran` of its `ng`.
  struct Cursor {
    int grp, b, hk, gran, ng, len;
    int id;                                        // the unit's number, where units are dealt out
  };
  Cursor c;                                        // start of the block's next piece
  int todo;                                        // places of the block's share of the list still to do
  const bool caller_splits = p.num_splits > 0;
  auto go_to_unit = [&](Cursor& x, int id) {       // (past the last unit: grp >= n_groups)
    x.id = id;
    x.hk = id % p.Hkv;
    x.b = id / p.Hkv % p.B;
    x.grp = id / p.Hkv / p.B;
    x.gran = 0;
    x.len = clamped_length(p, x.b);
    x.ng = granules_of(x.len);
  };
  bool by_units = p.by_units != 0;
  int rest = 0;                                    // places behind the granules of a unit
  // The block's place in the list, from the lengths; false: it has none.
  auto find_place = [&](int len0) -> bool {
    int before, all, longest;
    sum_granules(p, len0, 0, before, all, longest);
    const long long granules = (long long)all * p.Hkv * p.n_groups;
    by_units = dealt_by_units(DH, granules, (long long)p.n_groups * p.B * p.Hkv, longest, p.fit);
    rest = by_units ? 0 : unit_rest(DH, granules, p.fit);
    if (by_units) return true;
    const long long per_group = ((long long)all + (long long)p.B * rest) * p.Hkv, total = per_group * p.n_groups;
    const int n_shares = shares_for(DH, p.fit, p.max_shares, total);
    if (blockIdx.x >= n_shares) return false;
    const Dealt dealt(total, n_shares);
    long long at = dealt.begin(blockIdx.x);
    todo = int(dealt.size(blockIdx.x));
    c.id = 0;
    c.grp = int(div_places(at, per_group));
    at -= c.grp * per_group;                       // inside the group: find the sequence, 32 lengths at a time
    for (int b0 = 0;; b0 += 32) {
      const int len = b0 + lane < p.B ? clamp_length(p, b0 == 0 ? len0 : p.lengths[b0 + lane]) : 0;
      const int mine = len > 0 ? granules_of(len) + rest : 0;
      int upto = mine;
#pragma unroll
      for (int s = 1; s < 32; s <<= 1) {
        const int v = __shfl_up_sync(0xffffffffu, upto, s);
        if (lane >= s) upto += v;
      }
      const uint32_t hit = __ballot_sync(0xffffffffu, at < (long long)upto * p.Hkv);
      if (hit != 0u) {
        const int src = __ffs(hit) - 1;
        at -= (long long)__shfl_sync(0xffffffffu, upto - mine, src) * p.Hkv;
        c.b = b0 + src;
        c.len = __shfl_sync(0xffffffffu, len, src);
        break;
      }
      at -= (long long)__shfl_sync(0xffffffffu, upto, 31) * p.Hkv;
    }
    c.ng = granules_of(c.len);
    c.hk = int(at) / (c.ng + rest);                // (a sequence's places of all KV heads fit 32 bits)
    c.gran = int(at) % (c.ng + rest);
    return true;
  };
  bool placed = true;
  if (caller_splits || by_units) {
    grid_dep_wait();
  } else {
    int len0 = 0;
    for (bool behind = p.B > 32;; behind = true) {   // (one copy of the code: the second time it is in the instruction cache)
      if (behind) grid_dep_wait();
      const int now = early_length(p);
      if (behind && p.B <= 32 && __all_sync(0xffffffffu, now == len0)) break;
      len0 = now;
      placed = find_place(len0);
      if (behind) break;
    }
  }
  if (blockIdx.x == 0 && warp == 0) {
    for (int b = lane; b < p.B; b += 32)
      if (p.lengths[b] < 1 || p.lengths[b] > p.max_pages * p.page_size) atomicOr(&g_dec_status, 2);  // clamped length
  }
  if (!placed) return;
  if (caller_splits) {
    const int split = blockIdx.x % p.num_splits;
    go_to_unit(c, blockIdx.x / p.num_splits);
    const int per = (c.ng + p.num_splits - 1) / p.num_splits;
    c.gran = min(c.ng, split * per);
    todo = min(c.ng - c.gran, per);
  } else if (by_units) {
    go_to_unit(c, blockIdx.x);
    if (c.grp >= p.n_groups) return;
    todo = c.ng;
  }

  uint8_t* ring = dsmem + size_t(warp) * STAGES * STAGE_BYTES;
  const uint32_t ring_u32 = smem_u32(ring);

  auto next_unit = [&](Cursor& x) {
    x.gran = 0;
    if (++x.hk == p.Hkv) {
      x.hk = 0;
      if (++x.b == p.B) {
        x.b = 0;
        ++x.grp;
      }
      x.len = clamped_length(p, x.b);
      x.ng = granules_of(x.len);
    }
  };
  // The piece behind the one at x, of the `left` places of the block's share from x on; past the end: grp >= n_groups.
  auto next_piece = [&](Cursor& x, int& left) {
    left -= min(left, x.ng + rest - x.gran);
    if (left > 0) {
      next_unit(x);
    } else if (by_units && !caller_splits) {
      go_to_unit(x, x.id + gridDim.x);
      left = x.ng;
    } else {
      x.grp = p.n_groups;
    }
  };

  if (c.gran >= c.ng && !caller_splits) {          // the share begins behind the granules of a unit
    next_piece(c, todo);
    if (c.grp >= p.n_groups) return;
  }

  // ---- copies: a cursor of their own, STAGES - 1 of this warp's granules ahead of the arithmetic ----
  Cursor f = c;                                    // start of the piece the copies are in
  int f_todo = todo;                               // places of the share from there on
  int f_left;                                      // granules of the piece from this warp's next one on (<= 0: none)
  const int gran_per_page = p.page_size / GRAN;
  const uint8_t *kbase = nullptr, *vbase = nullptr;   // the group's pools
  const int32_t* bt = nullptr;                     // block-table entry of the page the next granule is in,
  int in_page = 0, f_tok = 0;                      // its place there, and its first token
  size_t page_elem = 0;                            // offset of this KV head's block of that page
  int stage_in = 0;
  auto enter_page = [&]() {
    const int page = min(max(*bt, 0), p.n_pages - 1);
    page_elem = (size_t(page) * p.Hkv + f.hk) * p.page_size;
  };
  auto enter_piece = [&]() {
    f_left = min(f_todo, f.ng - f.gran) - warp;
    if (f_left <= 0) return;
    const int gran = f.gran + warp, col = gran / gran_per_page;
    kbase = reinterpret_cast<const uint8_t*>(p.grp[f.grp].k_cache);
    vbase = reinterpret_cast<const uint8_t*>(p.grp[f.grp].v_cache);
    bt = p.block_table + size_t(f.b) * p.max_pages + col;
    in_page = gran - col * gran_per_page;
    f_tok = gran * GRAN;
    enter_page();
  };
  auto issue_next = [&]() {
    // find the piece that holds the next granule of this warp (pieces may be shorter than the block has warps)
    while (f_left <= 0 && f.grp < p.n_groups) {
      next_piece(f, f_todo);
      if (f.grp < p.n_groups) enter_piece();
    }
    if (f_left > 0) {
      const size_t at = (page_elem + size_t(in_page) * GRAN) * ROW_BYTES;
      const uint8_t* ksrc = kbase + at;
      const uint8_t* vsrc = vbase + at;
      const uint32_t dst = ring_u32 + stage_in * STAGE_BYTES;
#pragma unroll
      for (int i = 0; i < CP_PER_LANE; ++i) {
        const int idx = i * 32 + lane;          // 16-byte chunk index inside the contiguous granule
        const int row = idx / CHUNKS, chunk = idx % CHUNKS;
        const uint32_t off = ring_off<DH>(row, chunk);
        // Slots at or past the sequence length were never appended and may hold anything (a NaN there would
        // survive the zero probability in P V): they are filled with zeros instead of being read.
        const uint32_t nbytes = f_tok + row < f.len ? 16u : 0u;
        cp_async16(dst + off, ksrc + size_t(idx) * 16, nbytes);
        cp_async16(dst + TILE_BYTES + off, vsrc + size_t(idx) * 16, nbytes);
      }
      if (++stage_in == STAGES) stage_in = 0;
      f_left -= DEC_WARPS;
      f_tok += DEC_WARPS * GRAN;
      in_page += DEC_WARPS;
      if (in_page >= gran_per_page && f_left > 0) {
        const int pages = in_page / gran_per_page;
        bt += pages;
        in_page -= pages * gran_per_page;
        enter_page();
      }
    }
    cp_async_commit();
  };
  enter_piece();
  // query fragments (A operand, rows = members x heads of the group, zero beyond its rows); those of the next piece are
  // requested before the merge at the end of a piece
  uint32_t qa[KSTEPS][4];
  auto load_queries = [&]() {
    const DecGroup& grp = p.grp[c.grp];
    const int R = grp.n_members * G;
    const int r0 = g, r1 = g + 8;
    const size_t off0 = r0 < R ? (size_t(c.b) * p.Hq + c.hk * G + r0 % G) * DH : 0;
    const size_t off1 = r1 < R ? (size_t(c.b) * p.Hq + c.hk * G + r1 % G) * DH : 0;
    auto pair_at = [&](const void* base, size_t off, int col) -> uint32_t {   // two elements of a query row as bf16
      if (p.io_f32) {
        const float2 v = *reinterpret_cast<const float2*>(reinterpret_cast<const float*>(base) + off + col);
        return pack_bf16(v.x, v.y);
      }
      return *reinterpret_cast<const uint32_t*>(reinterpret_cast<const __nv_bfloat16*>(base) + off + col);
    };
    const void* q0 = r0 < R ? grp.q[r0 / G] : nullptr;
    const void* q1 = r1 < R ? grp.q[r1 / G] : nullptr;
#pragma unroll
    for (int ks = 0; ks < KSTEPS; ++ks) {
      const int col = ks * 16 + t * 2;
      qa[ks][0] = q0 ? pair_at(q0, off0, col) : 0u;
      qa[ks][1] = q1 ? pair_at(q1, off1, col) : 0u;
      qa[ks][2] = q0 ? pair_at(q0, off0, col + 8) : 0u;
      qa[ks][3] = q1 ? pair_at(q1, off1, col + 8) : 0u;
    }
  };

#pragma unroll
  for (int s = 0; s < STAGES - 1; ++s) issue_next();
  load_queries();

  int stage_out = 0;
  do {
    // ---- one unit, or this block's piece of it ----
    const DecGroup& grp = p.grp[c.grp];
    const int R = grp.n_members * G;               // valid query rows (<= 16)
    const int n_here = min(todo, c.ng - c.gran);
    const bool from_start = c.gran == 0, to_end = c.gran + n_here == c.ng;

    float oacc[NBLK][4];
#pragma unroll
    for (int n = 0; n < NBLK; ++n) oacc[n][0] = oacc[n][1] = oacc[n][2] = oacc[n][3] = 0.f;
    float m_run[2] = {-INFINITY, -INFINITY};  // rows g, g+8 (log2 domain)
    float l_run[2] = {0.f, 0.f};              // per-lane partial sums, against m_run
    float ref[2] = {-INFINITY, -INFINITY};    // reference of P and oacc

    for (int i = warp; i < n_here; i += DEC_WARPS) {
      cp_async_wait<STAGES - 2>();
      __syncwarp();
      issue_next();   // into the stage freed by the previous granule
      const int gran = c.gran + i;
      const uint32_t sK = ring_u32 + stage_out * STAGE_BYTES;
      const uint32_t sV = sK + TILE_BYTES;
      if (++stage_out == STAGES) stage_out = 0;

      // ---- S[16 rows, 16 tokens] = Q K^T ----
      float sacc[2][4];
#pragma unroll
      for (int nb = 0; nb < 2; ++nb) sacc[nb][0] = sacc[nb][1] = sacc[nb][2] = sacc[nb][3] = 0.f;
#pragma unroll
      for (int ks = 0; ks < KSTEPS; ++ks) {
        // four 8x8 matrices: (tokens 0-7, dh ks*16..+7), (tokens 0-7, +8..15), (tokens 8-15, ...), (tokens 8-15, +8)
        const int mat = lane >> 3, rr = lane & 7;
        const int row = (mat >> 1) * 8 + rr;
        const int chunk = ks * 2 + (mat & 1);
        uint32_t b00, b01, b10, b11;
        ldsm_x4(sK + ring_off<DH>(row, chunk), b00, b01, b10, b11);
        mma_bf16(sacc[0], qa[ks][0], qa[ks][1], qa[ks][2], qa[ks][3], b00, b01);
        mma_bf16(sacc[1], qa[ks][0], qa[ks][1], qa[ks][2], qa[ks][3], b10, b11);
      }
      // ---- online softmax over the 16 tokens ----
      const int tok0 = gran * GRAN;
      float mt[2] = {-INFINITY, -INFINITY};
#pragma unroll
      for (int nb = 0; nb < 2; ++nb) {
#pragma unroll
        for (int u = 0; u < 4; ++u) {
          const int tk = tok0 + nb * 8 + t * 2 + (u & 1);
          float x = sacc[nb][u] * p.scale_log2;
          if (tk >= c.len) x = -INFINITY;
          sacc[nb][u] = x;
          mt[u >> 1] = fmaxf(mt[u >> 1], x);
        }
      }
      const bool falls = (i / DEC_WARPS) % REFERENCE_GRANULES == 0;
      float alpha[2], beta[2], l_here[2] = {0.f, 0.f};
#pragma unroll
      for (int h = 0; h < 2; ++h) {
        mt[h] = fmaxf(mt[h], __shfl_xor_sync(0xffffffffu, mt[h], 1));
        mt[h] = fmaxf(mt[h], __shfl_xor_sync(0xffffffffu, mt[h], 2));
        const float m_new = fmaxf(m_run[h], mt[h]), ref_new = fmaxf(falls ? m_new - REFERENCE_DROP : ref[h], mt[h]);
        alpha[h] = ref[h] == -INFINITY ? 0.f : fast_exp2(ref[h] - ref_new);
        beta[h] = fast_exp2(ref_new - m_new);
        l_run[h] *= m_run[h] == -INFINITY ? 0.f : fast_exp2(m_run[h] - m_new);
        m_run[h] = m_new;
        ref[h] = ref_new;
      }
      uint32_t pa[4];
      {
        float pr[2][4];
#pragma unroll
        for (int nb = 0; nb < 2; ++nb)
#pragma unroll
          for (int u = 0; u < 4; ++u) {
            pr[nb][u] = fast_exp2(sacc[nb][u] - ref[u >> 1]);
            l_here[u >> 1] += pr[nb][u];
          }
#pragma unroll
        for (int h = 0; h < 2; ++h) l_run[h] = fmaf(l_here[h], beta[h], l_run[h]);
        pa[0] = pack_bf16(pr[0][0], pr[0][1]);
        pa[1] = pack_bf16(pr[0][2], pr[0][3]);
        pa[2] = pack_bf16(pr[1][0], pr[1][1]);
        pa[3] = pack_bf16(pr[1][2], pr[1][3]);
      }
      if (!__all_sync(0xffffffffu, alpha[0] == 1.f && alpha[1] == 1.f)) {
#pragma unroll
        for (int n = 0; n < NBLK; ++n) {
          oacc[n][0] *= alpha[0];
          oacc[n][1] *= alpha[0];
          oacc[n][2] *= alpha[1];
          oacc[n][3] *= alpha[1];
        }
      }
      // ---- O[16 rows, DH] += P[16 rows, 16 tokens] V[16 tokens, DH] ----
#pragma unroll
      for (int n2 = 0; n2 < NBLK / 2; ++n2) {
        // four 8x8 matrices (transposed on load): (tokens 0-7, dh n2*16..+7), (tokens 8-15, same dh),
        // (tokens 0-7, dh +8..15), (tokens 8-15, dh +8..15)
        const int mat = lane >> 3, rr = lane & 7;
        const int row = (mat & 1) * 8 + rr;
        const int chunk = n2 * 2 + (mat >> 1);
        uint32_t v00, v01, v10, v11;
        ldsm_x4_t(sV + ring_off<DH>(row, chunk), v00, v01, v10, v11);
        mma_bf16(oacc[2 * n2], pa[0], pa[1], pa[2], pa[3], v00, v01);
        mma_bf16(oacc[2 * n2 + 1], pa[0], pa[1], pa[2], pa[3], v10, v11);
      }
      __syncwarp();  // every lane is done with this stage before it is refilled
    }
    const Cursor here = c;
    next_piece(c, todo);
    const bool last = c.grp >= p.n_groups;
    if (last) grid_dep_launch();   // this warp's loads are out, the others' within a granule
    else load_queries();

#pragma unroll
    for (int h = 0; h < 2; ++h) {
      l_run[h] += __shfl_xor_sync(0xffffffffu, l_run[h], 1);
      l_run[h] += __shfl_xor_sync(0xffffffffu, l_run[h], 2);
      const float to_max = ref[h] == -INFINITY ? 1.f : fast_exp2(ref[h] - m_run[h]);   // at most 1
#pragma unroll
      for (int n = 0; n < NBLK; ++n) {
        oacc[n][2 * h] *= to_max;
        oacc[n][2 * h + 1] *= to_max;
      }
    }
    // ---- warp 0 merges the results of the others into its own, eight rows at a time ----
#pragma unroll
    for (int h = 0; h < 2; ++h) {
      if (8 * h >= R) break;
      __syncthreads();   // warp 0 is done with the previous ones
      if (warp > 0) {
#pragma unroll
        for (int n = 0; n < NBLK; ++n) s_o[warp - 1][n * 32 + lane] = make_float2(oacc[n][2 * h], oacc[n][2 * h + 1]);
        s_ml[warp - 1][lane] = make_float2(m_run[h], l_run[h]);
      }
      __syncthreads();
      if (warp == 0) {
        float2 om[DEC_WARPS - 1];
        float mn = m_run[h];
#pragma unroll
        for (int w = 0; w < DEC_WARPS - 1; ++w) {
          om[w] = s_ml[w][lane];
          mn = fmaxf(mn, om[w].x);
        }
        const float fa = m_run[h] == -INFINITY ? 0.f : fast_exp2(m_run[h] - mn);
        m_run[h] = mn;
        l_run[h] *= fa;
#pragma unroll
        for (int n = 0; n < NBLK; ++n) {
          oacc[n][2 * h] *= fa;
          oacc[n][2 * h + 1] *= fa;
        }
#pragma unroll
        for (int w = 0; w < DEC_WARPS - 1; ++w) {
          const float fb = om[w].x == -INFINITY ? 0.f : fast_exp2(om[w].x - mn);
          l_run[h] += om[w].y * fb;
#pragma unroll
          for (int n = 0; n < NBLK; ++n) {
            const float2 v = s_o[w][n * 32 + lane];
            oacc[n][2 * h] += v.x * fb;
            oacc[n][2 * h + 1] += v.y * fb;
          }
        }
      }
    }
    if (warp != 0) {
      // (warp 0 alone goes on to store)
    } else if (!caller_splits && from_start && to_end) {
      // ---- the whole unit: normalise and store ----
#pragma unroll
      for (int h = 0; h < 2; ++h) {
        const int row = g + 8 * h;
        if (row < R) {
          const int mem = row / G;
          const size_t head = size_t(here.b) * p.Hq + here.hk * G + row % G;
          const float inv = 1.f / l_run[h];
#pragma unroll
          for (int n = 0; n < NBLK; ++n) {
            const uint32_t v = pack_bf16(oacc[n][2 * h] * inv, oacc[n][2 * h + 1] * inv);   // rounded to bf16 either way: one set of results
            const size_t at = head * DH + n * 8 + t * 2;
            if (p.io_f32)
              *reinterpret_cast<float2*>(reinterpret_cast<float*>(grp.o[mem]) + at) = make_float2(__uint_as_float(v << 16), __uint_as_float(v & 0xffff0000u));
            else
              *reinterpret_cast<uint32_t*>(reinterpret_cast<__nv_bfloat16*>(grp.o[mem]) + at) = v;
          }
          if (t == 0) grp.lse[mem][head] = log_sum(m_run[h], l_run[h]);
        }
      }
    } else {
      // ---- a piece: the first of a share, or the last one if that starts a unit ----
      const size_t piece = caller_splits ? size_t(blockIdx.x) : size_t(blockIdx.x) * 2 + (from_start ? 1 : 0);
      float* po = p.part_o + piece * p.rows * DH;
      float* pml = p.part_ml + piece * p.rows * 2;
#pragma unroll
      for (int h = 0; h < 2; ++h) {
        const int row = g + 8 * h;
        if (row < R) {
#pragma unroll
          for (int n = 0; n < NBLK; ++n)
            *reinterpret_cast<float2*>(po + row * DH + n * 8 + t * 2) = make_float2(oacc[n][2 * h], oacc[n][2 * h + 1]);
          if (t == 0) *reinterpret_cast<float2*>(pml + row * 2) = make_float2(m_run[h], l_run[h]);
        }
      }
    }
    if (last) break;
  } while (true);
  cp_async_wait<0>();
}

// Merges the pieces of the units that more than one share holds and writes bf16 outputs and LSE.  Eight warps per block;
// `wpr` of them share a row of a unit (one where a unit has few pieces, eight where it has many), each lane four
// columns.  Bound: latency; the pieces are in L2.
constexpr int COMBINE_THREADS = 256;
template <int DH, int NG>
__global__ void __launch_bounds__(COMBINE_THREADS) decode_combine_kernel(const __grid_constant__ DecParams<NG> p, int wpr) {
  constexpr int LANES = DH / 4;               // lanes per piece and row
  constexpr int PER_WARP = 32 / LANES;        // pieces a warp takes at a time
  __shared__ float s_m[COMBINE_THREADS / 32], s_l[COMBINE_THREADS / 32];
  __shared__ float4 s_o[COMBINE_THREADS / 32][LANES];
  const int warp = threadIdx.x >> 5, lane = threadIdx.x & 31;
  const int rows_per_block = (COMBINE_THREADS / 32) / wpr;
  const int G = p.Hq / p.Hkv;
  const int unit = blockIdx.x;
  const int hk = unit % p.Hkv, b = unit / p.Hkv % p.B, gi = unit / p.Hkv / p.B;
  const DecGroup& grp = p.grp[gi];
  const int R = grp.n_members * G;
  const int row = blockIdx.y * rows_per_block + warp / wpr;
  grid_dep_launch();
  int w0 = 0, w1 = 0;                         // shares (or splits) that hold the unit
  if (p.num_splits > 0) {
    w0 = unit * p.num_splits;
    w1 = w0 + p.num_splits - 1;
    grid_dep_wait();
  } else {
    int len0 = 0;
    for (bool behind = p.B > 32;; behind = true) {
      if (behind) grid_dep_wait();
      const int now = early_length(p);
      if (behind && p.B <= 32 && __all_sync(0xffffffffu, now == len0)) break;
      len0 = now;
      int before, all, longest;
      sum_granules(p, len0, b, before, all, longest);
      const long long granules = (long long)all * p.Hkv * p.n_groups;
      if (dealt_by_units(DH, granules, (long long)p.n_groups * p.B * p.Hkv, longest, p.fit)) {
        w0 = w1 = 0;                          // finished by the blocks that held them
      } else {
        const int len = b < 32 ? __shfl_sync(0xffffffffu, len0, b) : p.lengths[b];
        const int rest = unit_rest(DH, granules, p.fit), ng = granules_of(clamp_length(p, len));
        const long long per_group = ((long long)all + (long long)p.B * rest) * p.Hkv, total = per_group * p.n_groups;
        const int n = shares_for(DH, p.fit, p.max_shares, total);
        const long long first = gi * per_group + ((long long)before + (long long)b * rest) * p.Hkv + (long long)hk * (ng + rest);
        const Dealt dealt(total, n);
        w0 = dealt.share_of(first);
        w1 = dealt.share_of(first + ng - 1);
      }
      if (behind) break;
    }
    if (w0 == w1) return;                     // finished by the block that had the share
  }
  if (blockIdx.y * rows_per_block >= R) return;
  const int sub = lane / LANES, col = (lane % LANES) * 4;
  float m = -INFINITY, l = 0.f;
  float4 acc = make_float4(0.f, 0.f, 0.f, 0.f);
  if (row < R) {
    constexpr int UNROLL = 4;                 // pieces in flight per lane
    const int step = wpr * PER_WARP;
    for (int w = w0 + (warp % wpr) * PER_WARP + sub; w <= w1; w += step * UNROLL) {
      float2 ml[UNROLL];
      float4 o[UNROLL];
#pragma unroll
      for (int u = 0; u < UNROLL; ++u) {
        const int wu = w + u * step;
        ml[u] = make_float2(-INFINITY, 0.f);
        if (wu <= w1) {
          const size_t piece = p.num_splits > 0 ? size_t(wu) : size_t(wu) * 2 + (wu == w0 ? 1 : 0);
          ml[u] = *reinterpret_cast<const float2*>(p.part_ml + (piece * p.rows + row) * 2);
          o[u] = *reinterpret_cast<const float4*>(p.part_o + (piece * p.rows + row) * DH + col);
        }
      }
#pragma unroll
      for (int u = 0; u < UNROLL; ++u) {
        if (ml[u].x == -INFINITY) continue;   // an empty split
        const float mn = fmaxf(m, ml[u].x);
        const float fa = m == -INFINITY ? 0.f : fast_exp2(m - mn), fb = fast_exp2(ml[u].x - mn);
        acc.x = acc.x * fa + o[u].x * fb;
        acc.y = acc.y * fa + o[u].y * fb;
        acc.z = acc.z * fa + o[u].z * fb;
        acc.w = acc.w * fa + o[u].w * fb;
        l = l * fa + ml[u].y * fb;
        m = mn;
      }
    }
  }
  auto merge = [&](float om, float ol, const float4& oo) {
    if (om == -INFINITY) return;
    const float mn = fmaxf(m, om);
    const float fa = m == -INFINITY ? 0.f : fast_exp2(m - mn), fb = fast_exp2(om - mn);
    acc.x = acc.x * fa + oo.x * fb;
    acc.y = acc.y * fa + oo.y * fb;
    acc.z = acc.z * fa + oo.z * fb;
    acc.w = acc.w * fa + oo.w * fb;
    l = l * fa + ol * fb;
    m = mn;
  };
  if (PER_WARP == 2) {                        // the two halves of the warp hold different pieces
    const float om = __shfl_xor_sync(0xffffffffu, m, 16), ol = __shfl_xor_sync(0xffffffffu, l, 16);
    const float4 oo = make_float4(__shfl_xor_sync(0xffffffffu, acc.x, 16), __shfl_xor_sync(0xffffffffu, acc.y, 16),
                                  __shfl_xor_sync(0xffffffffu, acc.z, 16), __shfl_xor_sync(0xffffffffu, acc.w, 16));
    merge(om, ol, oo);
  }
  if (wpr > 1) {                              // the block's warps hold pieces of one row (uniform: every thread arrives)
    if (lane < LANES) s_o[warp][lane] = acc;
    if (lane == 0) {
      s_m[warp] = m;
      s_l[warp] = l;
    }
    __syncthreads();
    if (warp % wpr != 0) return;
    for (int k = 1; k < wpr; ++k) merge(s_m[warp + k], s_l[warp + k], s_o[warp + k][lane % LANES]);
  }
  if (row < R && lane < LANES) {
    const int mem = row / G;
    const size_t head = size_t(b) * p.Hq + hk * G + row % G;
    const float inv = 1.f / l;
    const uint2 v = make_uint2(pack_bf16(acc.x * inv, acc.y * inv), pack_bf16(acc.z * inv, acc.w * inv));   // rounded to bf16 either way
    if (p.io_f32)
      *reinterpret_cast<float4*>(reinterpret_cast<float*>(grp.o[mem]) + head * DH + col) =
          make_float4(__uint_as_float(v.x << 16), __uint_as_float(v.x & 0xffff0000u), __uint_as_float(v.y << 16), __uint_as_float(v.y & 0xffff0000u));
    else
      *reinterpret_cast<uint2*>(reinterpret_cast<__nv_bfloat16*>(grp.o[mem]) + head * DH + col) = v;
    if (lane == 0) grp.lse[mem][head] = log_sum(m, l);
  }
}

// Owners write the new token's K and V rows into their pages.
struct AppendLayer {
  const void *k_new, *v_new;           // [B,Hkv,dh] bf16, or fp32 when new_f32 (rounded to bf16 as it is stored)
  __nv_bfloat16 *k_cache, *v_cache;
};
struct AppendSizes {
  const int32_t* block_table;
  const int32_t* lengths;
  int B, Hkv, dh, page_size, max_pages, n_pages;
  int new_f32;
};
template <int NG>
struct AppendParams : AppendSizes {
  AppendLayer at[NG];
};

template <int NG>
__global__ void append_kernel(const __grid_constant__ AppendParams<NG> p) {
  const int layer = blockIdx.y;
  const int b = blockIdx.x;
  grid_dep_launch();
  grid_dep_wait();
  const int row_chunks = p.dh / 8;  // 16-byte chunks per head row
  auto eight = [&](const void* base, int idx) -> uint4 {   // eight consecutive elements as bf16
    const size_t src = size_t(b) * p.Hkv * p.dh + size_t(idx) * 8;
    if (p.new_f32) {
      const float4 a = *reinterpret_cast<const float4*>(reinterpret_cast<const float*>(base) + src);
      const float4 c4 = *reinterpret_cast<const float4*>(reinterpret_cast<const float*>(base) + src + 4);
      return make_uint4(pack_bf16(a.x, a.y), pack_bf16(a.z, a.w), pack_bf16(c4.x, c4.y), pack_bf16(c4.z, c4.w));
    }
    return *reinterpret_cast<const uint4*>(reinterpret_cast<const __nv_bfloat16*>(base) + src);
  };
  // the new rows are asked for before the page is known, which takes two loads
  const int n = p.Hkv * row_chunks;
  uint4 k = make_uint4(0u, 0u, 0u, 0u), v = k;
  if (threadIdx.x < n) {
    k = eight(p.at[layer].k_new, threadIdx.x);
    v = eight(p.at[layer].v_new, threadIdx.x);
  }
  const int len = p.lengths[b];
  const int cap = p.max_pages * p.page_size;
  if (len < 1 || len > cap) return;  // nothing sensible to write; decode flags the bad length
  const int pos = len - 1;
  const int page = p.block_table[size_t(b) * p.max_pages + pos / p.page_size];
  if (page < 0 || page >= p.n_pages) return;
  for (int idx = threadIdx.x; idx < n;) {
    const int hk = idx / row_chunks, c = idx % row_chunks;
    const size_t dst = ((size_t(page) * p.Hkv + hk) * p.page_size + pos % p.page_size) * p.dh + c * 8;
    *reinterpret_cast<uint4*>(p.at[layer].k_cache + dst) = k;
    *reinterpret_cast<uint4*>(p.at[layer].v_cache + dst) = v;
    idx += blockDim.x;
    if (idx < n) {
      k = eight(p.at[layer].k_new, idx);
      v = eight(p.at[layer].v_new, idx);
    }
  }
}

template <int NG>
cudaError_t launch_append(const AppendParams<MAX_DEC_GROUPS>& all, int n, cudaStream_t stream) {
  AppendParams<NG> p;
  static_cast<AppendSizes&>(p) = all;
  std::copy(all.at, all.at + n, p.at);
  return launch_kernel(append_kernel<NG>, dim3(all.B, n), 128, 0, stream, 1, p);
}

int check_desc(const kvp_decode_desc* d) {
  if (d == nullptr) return KVP_ERR_INVALID_ARG;
  if (d->L < 1 || d->B < 1 || d->Hq < 1 || d->Hkv < 1 || d->max_pages < 1 || d->n_pages < 1 || d->num_splits < 0)
    return KVP_ERR_INVALID_ARG;
  if (d->dtype != KVP_BF16 && d->dtype != KVP_F32) return KVP_ERR_UNSUPPORTED;
  if ((d->dh != 64 && d->dh != 128) || d->Hq % d->Hkv != 0 || d->Hq / d->Hkv > 16 || d->page_size < GRAN ||
      d->page_size % GRAN != 0)
    return KVP_ERR_UNSUPPORTED;
  return KVP_OK;
}

// Sub-groups of at most min(MAX_MEMBERS, 16 / G) layers that share a donor inside [begin, end).
struct SubGroup {
  int owner;
  int members[MAX_MEMBERS];
  int n;
};

int build_groups(const kvp_decode_desc* d, const int32_t* donor, int begin, int end, SubGroup* out, int max_out) {
  const int G = d->Hq / d->Hkv;
  int per = 16 / G;
  if (per > MAX_MEMBERS) per = MAX_MEMBERS;
  int n_out = 0;
  for (int own = 0; own < d->L; ++own) {
    if (donor[own] != own) continue;
    SubGroup cur;
    cur.owner = own;
    cur.n = 0;
    for (int l = begin > own ? begin : own; l < end; ++l) {
      if (donor[l] != own) continue;
      cur.members[cur.n++] = l;
      if (cur.n == per) {
        if (n_out == max_out) return -1;
        out[n_out++] = cur;
        cur.n = 0;
      }
    }
    if (cur.n > 0) {
      if (n_out == max_out) return -1;
      out[n_out++] = cur;
    }
  }
  return n_out;
}

size_t align256(size_t x) { return (x + 255) & ~size_t(255); }

// Pieces and their bytes.  When the library chooses: two for each share of the list at its longest; with the
// caller's split count: one for every (unit, split).  One launch holds at most MAX_DEC_GROUPS sub-groups and launches
// reuse the space.
int blocks_that_fit(int dh) { return sm_count() * (dh == 128 ? DEC_CTAS_PER_SM<128> : DEC_CTAS_PER_SM<64>); }
size_t piece_bytes(const kvp_decode_desc* d, size_t pieces, int rows) {
  return align256(pieces * rows * d->dh * 4) + align256(pieces * rows * 2 * 4);
}
long long longest_unit(const kvp_decode_desc* d) { return (long long)d->max_pages * d->page_size / GRAN; }
long long longest_list(const kvp_decode_desc* d, int n_groups) { return (long long)n_groups * d->B * d->Hkv * longest_unit(d); }
struct Scratch {
  int max_shares = 0, rows = 0;
  size_t pieces = 0, bytes = 0;
};
// limit > 0: fewer shares until the pieces fit into that many bytes
Scratch plan_scratch(const kvp_decode_desc* d, const SubGroup* subs, int n_sub, size_t limit) {
  Scratch s;
  const int per_launch = n_sub < MAX_DEC_GROUPS ? n_sub : MAX_DEC_GROUPS;
  for (int i = 0; i < n_sub; ++i) s.rows = std::max(s.rows, subs[i].n * (d->Hq / d->Hkv));
  const int fit = blocks_that_fit(d->dh);
  const long long longest = longest_list(d, per_launch);
  s.max_shares = shares_for(d->dh, fit, fit * max_rounds(d->dh), longest + (long long)per_launch * d->B * d->Hkv * unit_rest(d->dh, longest, fit));
  for (;;) {
    s.pieces = d->num_splits > 0 ? size_t(per_launch) * d->B * d->Hkv * d->num_splits : size_t(s.max_shares) * 2;
    s.bytes = piece_bytes(d, s.pieces, s.rows);
    if (limit == 0 || s.bytes <= limit || d->num_splits > 0 || s.max_shares == 1) return s;
    s.max_shares = (s.max_shares + 1) / 2;
  }
}
// bytes for decoding layers [begin, end); 0 when the request cannot be served at all
size_t decode_scratch_bytes(const kvp_decode_desc* d, const int32_t* donor, int begin, int end) {
  static thread_local SubGroup tmp[4096];
  const int n_sub = build_groups(d, donor, begin, end, tmp, 4096);
  return n_sub <= 0 ? 0 : plan_scratch(d, tmp, n_sub, 0).bytes;
}

int decode_impl(const kvp_decode_desc* d, const int32_t* donor, float scale, const void* const* q, const void* const* k_cache,
                const void* const* v_cache, const int32_t* block_table, const int32_t* lengths, void* const* o,
                float* const* lse, int layer_begin, int layer_end, void* ws, size_t ws_bytes, size_t limit,
                cudaStream_t stream);

}  // namespace

int decode_read_status() {
  int v = 0;
  if (cudaMemcpyFromSymbol(&v, g_dec_status, sizeof(int)) != cudaSuccess) return -1;
  if (v != 0) {
    int zero = 0;
    cudaMemcpyToSymbol(g_dec_status, &zero, sizeof(int));
  }
  return v & 1;  // bit 1 (clamped length) is informational
}

}  // namespace kvp

using namespace kvp;

extern "C" size_t kvp_decode_workspace_bytes(const kvp_decode_desc* d, const int32_t* donor) {
  if (check_desc(d) != KVP_OK || donor == nullptr) return 0;
  return decode_scratch_bytes(d, donor, 0, d->L);
}

extern "C" int kvp_cache_append(const kvp_decode_desc* d, const int32_t* donor, const void* const* k_new,
                                const void* const* v_new, void* const* k_cache, void* const* v_cache,
                                const int32_t* block_table, const int32_t* lengths, kvp_stream_t stream_) {
  int rc = check_desc(d);
  if (rc != KVP_OK) return rc;
  if (donor == nullptr || k_new == nullptr || v_new == nullptr || k_cache == nullptr || v_cache == nullptr ||
      block_table == nullptr || lengths == nullptr)
    return KVP_ERR_INVALID_ARG;
  for (int l = 0; l < d->L; ++l)
    if (donor[l] < 0 || donor[l] > l || donor[donor[l]] != donor[l]) return KVP_ERR_BAD_DONOR;
  cudaStream_t stream = reinterpret_cast<cudaStream_t>(stream_);
  AppendParams<MAX_DEC_GROUPS> p;
  p.block_table = block_table;
  p.lengths = lengths;
  p.B = d->B;
  p.Hkv = d->Hkv;
  p.dh = d->dh;
  p.page_size = d->page_size;
  p.max_pages = d->max_pages;
  p.n_pages = d->n_pages;
  p.new_f32 = d->dtype == KVP_F32;
  int n = 0;
  for (int l = 0; l <= d->L; ++l) {
    const bool owner = l < d->L && donor[l] == l;  // consumers store nothing (Eq. 3)
    if (owner) {
      if (k_new[l] == nullptr || v_new[l] == nullptr || k_cache[l] == nullptr || v_cache[l] == nullptr)
        return KVP_ERR_INVALID_ARG;
      p.at[n++] = AppendLayer{k_new[l], v_new[l], reinterpret_cast<__nv_bfloat16*>(k_cache[l]), reinterpret_cast<__nv_bfloat16*>(v_cache[l])};
    }
    if (n == MAX_DEC_GROUPS || (l == d->L && n > 0)) {
      if ((n <= FEW_DEC_GROUPS ? launch_append<FEW_DEC_GROUPS>(p, n, stream) : launch_append<MAX_DEC_GROUPS>(p, n, stream)) != cudaSuccess) return KVP_ERR_CUDA;
      n = 0;
    }
  }
  return KVP_OK;
}

namespace kvp {
namespace {

template <int DH, int NG>
cudaError_t launch_decode(const DecParams<MAX_DEC_GROUPS>& all, dim3 grid, dim3 combine_grid, int wpr, cudaStream_t stream) {
  constexpr int smem = DEC_WARPS * DEC_STAGES * 2 * GRAN * DH * 2;
  cudaError_t e = allow_smem<decode_kernel<DH, NG>>(smem);
  if (e != cudaSuccess) return e;
  DecParams<NG> p;
  static_cast<DecSizes&>(p) = all;
  std::copy(all.grp, all.grp + all.n_groups, p.grp);
  timing_before(KVP_KERNEL_DECODE, stream);
  e = launch_kernel(decode_kernel<DH, NG>, grid, DEC_THREADS, smem, stream, 1, p);
  timing_after(KVP_KERNEL_DECODE, stream);
  if (e == cudaSuccess && (p.num_splits > 0 || p.by_units == 0))   // whole units leave no pieces
    e = launch_kernel(decode_combine_kernel<DH, NG>, combine_grid, COMBINE_THREADS, 0, stream, 1, p, wpr);
  return e;
}

int decode_impl(const kvp_decode_desc* d, const int32_t* donor, float scale, const void* const* q, const void* const* k_cache,
                const void* const* v_cache, const int32_t* block_table, const int32_t* lengths, void* const* o,
                float* const* lse, int layer_begin, int layer_end, void* ws, size_t ws_bytes, size_t limit,
                cudaStream_t stream) {
  int rc = check_desc(d);
  if (rc != KVP_OK) return rc;
  if (donor == nullptr || q == nullptr || k_cache == nullptr || v_cache == nullptr || block_table == nullptr ||
      lengths == nullptr || o == nullptr || lse == nullptr || scale < 0.f)
    return KVP_ERR_INVALID_ARG;
  if (layer_begin < 0 || layer_end > d->L || layer_begin >= layer_end) return KVP_ERR_INVALID_ARG;
  for (int l = 0; l < d->L; ++l)
    if (donor[l] < 0 || donor[l] > l || donor[donor[l]] != donor[l]) return KVP_ERR_BAD_DONOR;
  static thread_local SubGroup subs[4096];
  const int n_sub = build_groups(d, donor, layer_begin, layer_end, subs, 4096);
  if (n_sub < 0) return KVP_ERR_UNSUPPORTED;
  const Scratch sc_plan = plan_scratch(d, subs, n_sub, limit);
  if (ws == nullptr || ws_bytes < sc_plan.bytes || !aligned16(ws)) return KVP_ERR_WORKSPACE;
  const size_t po_bytes = align256(sc_plan.pieces * sc_plan.rows * d->dh * 4);

  DecParams<MAX_DEC_GROUPS> p;
  p.block_table = block_table;
  p.lengths = lengths;
  p.part_o = reinterpret_cast<float*>(ws);
  p.part_ml = reinterpret_cast<float*>(reinterpret_cast<uint8_t*>(ws) + po_bytes);
  p.B = d->B;
  p.Hq = d->Hq;
  p.Hkv = d->Hkv;
  p.page_size = d->page_size;
  p.max_pages = d->max_pages;
  p.n_pages = d->n_pages;
  p.rows = sc_plan.rows;
  p.fit = blocks_that_fit(d->dh);
  p.max_shares = sc_plan.max_shares;
  p.num_splits = d->num_splits;
  p.io_f32 = d->dtype == KVP_F32;
  const float sc = scale == 0.f ? 1.f / sqrtf(float(d->dh)) : scale;
  p.scale_log2 = sc * 1.4426950408889634f;

  for (int s0 = 0; s0 < n_sub; s0 += MAX_DEC_GROUPS) {
    const int n = n_sub - s0 < MAX_DEC_GROUPS ? n_sub - s0 : MAX_DEC_GROUPS;
    int rows = 0;
    for (int i = 0; i < n; ++i) {
      const SubGroup& sg = subs[s0 + i];
      DecGroup& g = p.grp[i];
      if (k_cache[sg.owner] == nullptr || v_cache[sg.owner] == nullptr) return KVP_ERR_INVALID_ARG;
      g.k_cache = reinterpret_cast<const __nv_bfloat16*>(k_cache[sg.owner]);
      g.v_cache = reinterpret_cast<const __nv_bfloat16*>(v_cache[sg.owner]);
      g.n_members = sg.n;
      g.pad = 0;
      rows = std::max(rows, sg.n * (d->Hq / d->Hkv));
      for (int m = 0; m < MAX_MEMBERS; ++m) {
        const int l = sg.members[m < sg.n ? m : 0];
        if (q[l] == nullptr || o[l] == nullptr || lse[l] == nullptr) return KVP_ERR_INVALID_ARG;
        g.q[m] = q[l];
        g.o[m] = o[l];
        g.lse[m] = lse[l];
      }
    }
    const long long units = (long long)n * d->B * d->Hkv;
    // a block for every share of the longest list; shares go by the lengths on the device, and so does whether whole units
    // are dealt out instead
    const long long blocks = d->num_splits > 0 ? units * d->num_splits
                                               : std::max((long long)sc_plan.max_shares, std::min(units, (long long)p.fit * max_rounds(d->dh)));
    if (units > 0x7fffffffLL || blocks > 0x7fffffffLL) return KVP_ERR_UNSUPPORTED;
    p.n_groups = n;
    // (units that are short on average in a full table are so at any lengths)
    p.by_units = dealt_by_units(d->dh, longest_list(d, n), units, longest_unit(d), p.fit);
    const long long unit_pieces = d->num_splits > 0 ? d->num_splits : sc_plan.max_shares / units;
    const int wpr = unit_pieces > 8 ? 8 : 1;   // many pieces a unit: eight warps share those of a row
    const int rows_per_block = COMBINE_THREADS / 32 / wpr;
    const dim3 grid(static_cast<unsigned>(blocks));
    const dim3 cgrid(unsigned(units), (rows + rows_per_block - 1) / rows_per_block);
    const bool few = n <= FEW_DEC_GROUPS;
    const cudaError_t e = d->dh == 128 ? (few ? launch_decode<128, FEW_DEC_GROUPS>(p, grid, cgrid, wpr, stream) : launch_decode<128, MAX_DEC_GROUPS>(p, grid, cgrid, wpr, stream))
                                       : (few ? launch_decode<64, FEW_DEC_GROUPS>(p, grid, cgrid, wpr, stream) : launch_decode<64, MAX_DEC_GROUPS>(p, grid, cgrid, wpr, stream));
    if (e != cudaSuccess) return KVP_ERR_CUDA;
  }
  return KVP_OK;
}

}  // namespace
}  // namespace kvp

extern "C" int kvp_decode(const kvp_decode_desc* d, const int32_t* donor, float scale, const void* const* q,
                          const void* const* k_cache, const void* const* v_cache, const int32_t* block_table,
                          const int32_t* lengths, void* const* o, float* const* lse, int layer_begin, int layer_end,
                          void* ws, size_t ws_bytes, kvp_stream_t stream) {
  return decode_impl(d, donor, scale, q, k_cache, v_cache, block_table, lengths, o, lse, layer_begin, layer_end, ws,
                     ws_bytes, 0, reinterpret_cast<cudaStream_t>(stream));
}

// ---------------------------------------------------------------------------------------------
// Decode without any caller-provided or allocated scratch.
//
// Some callers cannot allocate device memory at the point where they decode: a serving loop that
// has handed the whole device to its own cache pool and has nothing left to carve a workspace
// from, a plug-in running inside a host application that forbids cudaMalloc on its hot path, or a
// worker that must not touch the allocator because another thread holds it.  For them the per-split
// partial results live in a fixed array that is part of the library image.
// ---------------------------------------------------------------------------------------------
namespace kvp {
namespace {

static __device__ __align__(256) unsigned char g_decode_scratch[KVP_DECODE_STATIC_SCRATCH_BYTES];

constexpr int kMaxDevices = 64;
std::mutex g_scratch_mutex;
void* g_scratch_ptr[kMaxDevices] = {};  // device address of g_decode_scratch, per device ordinal

// The array's name is only a host-side handle here; kernels need its device address, which differs
// per device and is looked up once with that device current.
int static_scratch_address(void** out) {
  int dev = -1;
  if (cudaGetDevice(&dev) != cudaSuccess || dev < 0 || dev >= kMaxDevices) return KVP_ERR_CUDA;
  std::lock_guard<std::mutex> lock(g_scratch_mutex);
  if (g_scratch_ptr[dev] == nullptr) {
    void* p = nullptr;
    if (cudaGetSymbolAddress(&p, g_decode_scratch) != cudaSuccess || p == nullptr) return KVP_ERR_CUDA;
    g_scratch_ptr[dev] = p;
  }
  *out = g_scratch_ptr[dev];
  return KVP_OK;
}

}  // namespace
}  // namespace kvp

extern "C" int kvp_decode_static(const kvp_decode_desc* d, const int32_t* donor, float scale, const void* const* q,
                                 const void* const* k_cache, const void* const* v_cache, const int32_t* block_table,
                                 const int32_t* lengths, void* const* o, float* const* lse, int layer_begin,
                                 int layer_end, kvp_stream_t stream) {
  int rc = check_desc(d);
  if (rc != KVP_OK) return rc;
  if (donor == nullptr) return KVP_ERR_INVALID_ARG;
  for (int l = 0; l < d->L; ++l)
    if (donor[l] < 0 || donor[l] > l || donor[donor[l]] != donor[l]) return KVP_ERR_BAD_DONOR;
  if (layer_begin < 0 || layer_end > d->L || layer_begin >= layer_end) return KVP_ERR_INVALID_ARG;
  // only the donor groups that the layer range touches need room, so a narrower range can fit where all layers do not
  // (when the library deals the rows out, it does so in fewer shares until their pieces fit)
  const size_t need = decode_scratch_bytes(d, donor, layer_begin, layer_end);
  if (need == 0) return KVP_ERR_UNSUPPORTED;
  if (d->num_splits > 0 && need > size_t(KVP_DECODE_STATIC_SCRATCH_BYTES)) return KVP_ERR_STATIC_SCRATCH;
  void* scratch = nullptr;
  rc = static_scratch_address(&scratch);
  if (rc != KVP_OK) return rc;
  return decode_impl(d, donor, scale, q, k_cache, v_cache, block_table, lengths, o, lse, layer_begin, layer_end, scratch,
                     size_t(KVP_DECODE_STATIC_SCRATCH_BYTES), size_t(KVP_DECODE_STATIC_SCRATCH_BYTES),
                     reinterpret_cast<cudaStream_t>(stream));
}
