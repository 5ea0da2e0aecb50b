// Fused block scoring and selection (Eq. 19, Eq. 20; Algorithm 1 lines 3-5) for plans whose packed query tiles come
// as TMA boxes (DevParams::q_box): score_select_kernel with TWO adjacent query tiles of a KV head per unit.
//
// At long sequences score_select_kernel is bound by the traffic of the pooled keys from L2 into shared memory: every
// chunk of 128 pooled keys (hi + lo: 64 KB) is fetched once per query tile, 35 bytes per cycle and SM at 131072
// tokens, before the tensor pipe (1024 cycles per chunk) or the exponentials (1024) are busy.  Adjacent tiles of one
// KV head have the same candidates (the later one at most one block more), so here a chunk of pooled keys, once in
// shared memory, is multiplied with both tiles in one MMA of N = 256 (A = 128 pooled keys on the TMEM lanes,
// B = the two query tiles back to back): half the bytes per tile, half the MMA instructions.
//
// Units (built by the planner, heaviest first): a pair of tiles (t-1, t) of one (sequence, KV head) when the later
// tile has at most 1024 candidate blocks, else a single tile.  CTA b takes units b, b + grid, b + 2 grid, ...
// As in score_select_kernel the contraction runs transposed and kbar enters as a 16-bit (hi, lo) pair accumulated into one fp32
// accumulator; per pooled key a consumer thread takes maximum and exponential sum over a tile's rows, log2 energies go to
// shared memory, and a selection warp applies threshold and forced sets and writes the ordered lists of unit u beside the
// scoring of unit u+1.
//
// What bounds it: per chunk of a pair the tensor pipe needs 2048 cycles and the exponentials 2048 of the MUFU pipe; measured
// about 2700 at the clocks that the power limit leaves at 131072 tokens (without the exponentials 7 % less, without the MMAs
// the same).  The items (chunk, tile) are dealt to THREE consumer warpgroups, so that one loads or waits while the others
// exponentiate, and an item goes through in batches (see score_cols), which is what lets three of them fit into the registers.
// Whole calls, two warpgroups with a tile each and 128 columns in one piece / so: lists of 65536 tokens 398 / 390 us, of 22965
// 115.0 / 112.5; attention included 131072 tokens 10828 / 10790.  FP8 plans took one tile per chunk in score_select_kernel before:
// 131072 tokens, 28 heads on 4, 7935 / 7720, 16 sequences 3492 / 3357, 8191 tokens 204.7 / 200.6.
//
// FP8: the raw e4m3 box lands in the second half of a query buffer, where its 128-byte rows are as many as the F16 rows of a
// half, and the consumer warps widen it in place, one unit ahead: elements 0..63 of a row go to the first half, 64..127 over the
// raw row.  Every row has a multiplier of its own (q_scale), kept per unit in sC.  One warp that fetched and widened the tiles was
// what the units waited for (8191 tokens, one chunk of keys per unit: 8900 cycles a unit, of which 5000 widening and 2100 the box).
// Select call in us, widened by one warp / by the consumers: 8191 tokens, 28 heads on 4, 42.6 / 32.8, 12000 tokens, 32 on 8, 66.8 /
// 48.8; lists of 12000 tokens with export 77.0 / 57.8 (row multipliers in registers on both sides); with attention 16 sequences
// 3222 / 3186, 131072 tokens the same.
//
// Roles: warps 0-11 consumers; warp 12 TMA producer of kbar pieces (16 KB: 128 keys x 64 elements, four per chunk: hi | lo x
// the two halves of d); warp 13 UMMA issuer and TMEM owner; warp 14 unit set-up and query tiles by TMA (two units in flight);
// warp 15 selection.
// Shared memory: 2 x 64 KB query pairs (and 5 KB of padding each) + 4 x 16 KB pieces + 16 KB energies.  TMEM: 2 x 256
// columns.
//
// Group sizes that do not divide 128 (7 and the like) used to stage every tile with 2048 cp.async pieces of 16 bytes, each
// with its own divisions: select + sparse of 24 sequences of 60 to 1500 tokens, 28 query heads on 4 KV heads, 360 us then, 170
// with the boxes in this kernel and the attention kernel.
#pragma once
#include "score_select.cuh"

namespace fp2 {

constexpr int kPairGroups = 3;           // consumer warpgroups
constexpr int kPairConsumers = kPairGroups * 128;
constexpr int kPairThreads = kPairConsumers + 128;
constexpr int kPairInfoSlots = 4;        // unit descriptors in flight
constexpr int kPairQBufs = 2;            // 64 KB query-pair buffers
constexpr int kPairPieces = 4;           // ring of 16 KB kbar pieces
constexpr int kPairPieceBytes = 16384;
constexpr int kPairMaxCand = 1024;       // a tile is paired only if it has at most this many candidate blocks
constexpr int kPairQHalf = 32768 + kQTailRows * 128;                // 256 rows x 128 bytes and the overhang behind them
constexpr int kPairQBytes = kQLeadRows * 128 + 2 * kPairQHalf;      // (the overhang in front of the second half falls there too)
static_assert(kQLeadRows * 128 % 1024 == 0 && kPairQHalf % 1024 == 0, "query halves start on the swizzle's period");
constexpr int kPairSmemBytes = 1024 /*align*/ + kPairQBufs * kPairQBytes + kPairPieces * kPairPieceBytes + kMaxBlocks * 4;

struct PairInfo {
  SegInfo sg[2];
  int32_t nt;       // tiles in the unit: 1 or 2
  int32_t valid;    // 0: no more work
};

// One pooled key (= this thread's TMEM lane) against the 128 query rows of one tile (= 128 TMEM columns at
// lane_addr): returns log2 sum_j 2^x_j, x_j = s_j * cs (FP8: s_j * sC[j]).  PARTIAL: only the first nrows columns are real
// query rows.  The columns go through in batches of W.  The reference of the exponentials is the maximum of the first 16
// columns instead of all 128 (no need to hold 128 logits, an eighth of the maxima): the sum is then at least 1, so nothing
// that matters underflows, and a batch after which it comes near the top of fp32 is done again with its own maximum.  The
// reference is kept finite: where the first 16 logits are all below the range of fp32 (-inf; queries of -3e38 will do) the
// others count as ever.  A key whose logits are all -inf has no energy: NaN, which no threshold keeps.  The accumulator is
// handed back once the last batch is in registers.
template <bool FP8, int NP, bool PARTIAL>
__device__ __forceinline__ float score_cols(uint32_t lane_addr, float cs, const float* sC, int nrows, uint64_t* release) {
  uint64_t period[NP > 0 ? NP : 1];
#pragma unroll
  for (int k = 0; k < NP; ++k) period[k] = reinterpret_cast<const uint64_t*>(sC)[k];
  constexpr int W = FP8 && NP == 0 ? 32 : 64;   // multipliers from shared memory take registers too: with 64 columns they spill (131072 tokens 1010 -> 1590 us)
  constexpr int kFirst = 16;
  float m = -INFINITY, total = 0.f;
  uint64_t s4[4] = {0ull, 0ull, 0ull, 0ull};   // sums of 2^(x_j - m), four independent (lo, hi) accumulators
#pragma unroll
  for (int j0 = 0; j0 < kTileRows; j0 += W) {
    uint32_t xv[W];
#pragma unroll
    for (int k = 0; k < W; k += 32) tmem_ld32(lane_addr + j0 + k, reinterpret_cast<uint32_t(&)[32]>(xv[k]));
#pragma unroll
    for (int k = 0; k < W; k += 32) tmem_wait_ld32(reinterpret_cast<uint32_t(&)[32]>(xv[k]));
    if (j0 + W == kTileRows) {
      tc_fence_before();
      mbar_arrive(release);
    }
    auto mult2 = [&](int j) {
      if constexpr (!FP8) return f2_pack(cs, cs);
      else if constexpr (NP > 0) return period[((j0 + j) >> 1) % NP];
      else return *reinterpret_cast<const uint64_t*>(sC + j0 + j);
    };
    auto batch_max = [&](int n) {   // of the first n scaled logits
      float mx[4] = {-INFINITY, -INFINITY, -INFINITY, -INFINITY};
#pragma unroll
      for (int j = 0; j < n; j += 2) {
        float a, c;
        if constexpr (FP8) {
          f2_unpack(f2_mul(f2_pack(__uint_as_float(xv[j]), __uint_as_float(xv[j + 1])), mult2(j)), a, c);
        } else {   // the multiplier is positive: it commutes with the maximum
          a = __uint_as_float(xv[j]);
          c = __uint_as_float(xv[j + 1]);
        }
        if constexpr (PARTIAL) {
          a = j0 + j < nrows ? a : -INFINITY;
          c = j0 + j + 1 < nrows ? c : -INFINITY;
        }
        mx[(j >> 1) & 3] = max3(mx[(j >> 1) & 3], a, c);
      }
      const float r = fmaxf(max3(mx[0], mx[1], mx[2]), mx[3]);
      return FP8 ? r : r * cs;
    };
    auto add_batch = [&]() {
      const uint64_t nm2 = f2_pack(-m, -m);
#pragma unroll
      for (int j = 0; j < W; j += 2) {
        float d0, d1;
        f2_unpack(f2_fma(f2_pack(__uint_as_float(xv[j]), __uint_as_float(xv[j + 1])), mult2(j), nm2), d0, d1);
        if constexpr (PARTIAL) {
          d0 = j0 + j < nrows ? d0 : -INFINITY;
          d1 = j0 + j + 1 < nrows ? d1 : -INFINITY;
        }
        s4[(j >> 1) & 3] = f2_add(s4[(j >> 1) & 3], f2_pack(ex2(d0), ex2(d1)));
      }
      float t0, t1;
      f2_unpack(f2_add(f2_add(s4[0], s4[1]), f2_add(s4[2], s4[3])), t0, t1);
      return t0 + t1;
    };
    if (j0 == 0) m = fmaxf(batch_max(kFirst), -3.402823466e38f);
    float sum = add_batch();
    if (__any_sync(0xffffffffu, sum > 1e36f)) {   // (as one warp: the next batch's TMEM loads want it whole)
      const float m_new = fmaxf(m, batch_max(W));
      s4[0] = f2_pack(total * ex2(m - m_new), 0.f);   // (total = 0 in the first batch, m is finite)
      s4[1] = s4[2] = s4[3] = 0ull;
      m = m_new;
      sum = add_batch();
    }
    total = sum;
  }
  return total > 0.f ? m + log2f(total) : __int_as_float(0x7fc00000);
}

// Raw e4m3 rows in the second half of a query buffer -> F16 rows in both halves, in place; by all consumer warps, four rows of
// 128 bytes per warp and step.  Eight lanes take a row; a warp's rows are in registers before the first of them is overwritten.
// The conversion runs at an eighth of the issue rate, on the pipe of the exponentials: 512 warp instructions for a pair, 1024
// cycles of each scheduler's, half of what the exponentials of one chunk take, once per unit.  Where a unit has one chunk or two that
// is a good part of it.
__device__ __forceinline__ void widen_pair_in_place(uint8_t* half0, uint8_t* half1, int rows, int warp, int lane) {
  constexpr int kStep = 16 * kPairGroups;   // rows per step
  const int c = lane & 7;
  uint8_t* const half = c < 4 ? half0 : half1;
#pragma unroll 1
  for (int row0 = warp * 4 + (lane >> 3); row0 - (lane >> 3) < rows; row0 += 2 * kStep) {
    uint4 v[2];
#pragma unroll
    for (int u = 0; u < 2; ++u)
      if (row0 + u * kStep < rows) v[u] = *reinterpret_cast<const uint4*>(half1 + sw128_offset(row0 + u * kStep, c));
    __syncwarp();
#pragma unroll
    for (int u = 0; u < 2; ++u)
      if (row0 + u * kStep < rows) {
        const int row = row0 + u * kStep;
        *reinterpret_cast<uint4*>(half + sw128_offset(row, (c & 3) * 2)) =
            make_uint4(e4m3x2_to_f16x2(v[u].x), e4m3x2_to_f16x2(v[u].x >> 16), e4m3x2_to_f16x2(v[u].y),
                       e4m3x2_to_f16x2(v[u].y >> 16));
        *reinterpret_cast<uint4*>(half + sw128_offset(row, (c & 3) * 2 + 1)) =
            make_uint4(e4m3x2_to_f16x2(v[u].z), e4m3x2_to_f16x2(v[u].z >> 16), e4m3x2_to_f16x2(v[u].w),
                       e4m3x2_to_f16x2(v[u].w >> 16));
      }
  }
}

// NP: FP8 plans whose heads repeat every NP pairs of rows of a tile hold the row multipliers in registers, NP pairs: 4 (group sizes
// that divide 8), 3 (3, 6), 5 (5, 10), 7 (7); 0: read from shared memory (9, 16 and more; more pairs would take registers that the
// columns need).  Read for every pair of columns they are a load each, which waits behind the operands of the MMAs, and leave no
// room for batches of 64 columns.  The registers are full: NP 3 and 4 spill 4 and 12 bytes, 5 and 7 12 and 16; with batches of 32
// nothing spills.  Lists and export of FP8 calls in us, in turn, from shared memory / registers and 32 columns / and 64: 12000
// tokens, groups of 3, 4, 5, 6 and 7: 54.2 / 51.9 / 50.8, 63.0 / 60.6 / 57.9, 74.9 / 72.1 / 67.8, 49.7 / 48.1 / 47.3, 55.0 / 53.2 / 51.3; 65536
// tokens 339 / 324 / 318, 435 / 417 / 406, 527 / 501 / 487, 314 / 301 / 296, 352 / 336 / 334.  Select + sparse of 16 sequences, groups of
// 4, 3273 / 3233 / 3211, 131072 tokens, groups of 7, 7644 / 7611 / 7602, 8191 tokens 174.0 / 172.3 / 172.0.
template <bool FP8, int NP>
__global__ void __launch_bounds__(kPairThreads, 1)
score_pair_kernel(const __grid_constant__ CUtensorMap map_khi, const __grid_constant__ CUtensorMap map_klo,
                  const __grid_constant__ CUtensorMap map_q, const __grid_constant__ CUtensorMap map_q2,
                  const SegInfo* __restrict__ segs, const int2* __restrict__ units, int nunits, const float* q_scale,
                  DevParams P, int64_t* __restrict__ seg_offset, int32_t* __restrict__ seg_count,
                  int32_t* __restrict__ blk_idx, int* __restrict__ status) {
  extern __shared__ uint8_t smem_raw[];
  uint8_t* smem = reinterpret_cast<uint8_t*>((reinterpret_cast<uintptr_t>(smem_raw) + 1023) & ~uintptr_t(1023));
  // query pair buffer: [half of d][tile][128 rows x 128 bytes] -- the two tiles of a half are 256 consecutive packed rows,
  // one swizzled K-major operand and one TMA box
  uint8_t* sQ = smem + kQLeadRows * 128;
  uint8_t* sStage = smem + kPairQBufs * kPairQBytes;                                  // ring of kbar pieces
  float* sE = reinterpret_cast<float*>(sStage + kPairPieces * kPairPieceBytes); // log2 energies: unit parity x 2048,
                                                                                // second tile of a pair 1024 further

  __shared__ PairInfo info[kPairInfoSlots];
  __shared__ __align__(8) float sC[FP8 ? kPairInfoSlots : 1][FP8 ? 2 * kTileRows : 2];   // per-row multipliers of the unit; rewritten
                                                                            // once the consumers have released the descriptor
  __shared__ uint64_t info_full[kPairInfoSlots], info_empty[kPairInfoSlots], q_full[kPairQBufs], q_empty[kPairQBufs];
  __shared__ uint64_t raw_full[kPairQBufs];
  __shared__ uint64_t full[kPairPieces], empty[kPairPieces], acc_full[2], acc_empty[2];
  __shared__ uint64_t e_full[2], sel_done[2];   // [unit & 1] energies of the unit are complete / its lists are written
  __shared__ uint64_t drain_bar;
  __shared__ uint32_t tmem_base_s;
  __shared__ int abort_flag;
  __shared__ float red[2][2][4 * kPairGroups];                // [unit & 1][tile][consumer warp] maxima of the log2 energies

  const int tid = threadIdx.x, warp = tid >> 5, lane = tid & 31;
  WaitCtx ctx{status, &abort_flag};

  if (tid == 0) {
    abort_flag = 0;
    for (int i = 0; i < kPairInfoSlots; ++i) {
      mbar_init(&info_full[i], 1);
      mbar_init(&info_empty[i], 2 + kPairConsumers + 1);   // producer, issuer, consumers, selection warp
    }
    for (int i = 0; i < kPairQBufs; ++i) {
      mbar_init(&q_full[i], FP8 ? 4 * kPairGroups : 1);   // FP8: the consumer warps, which widen the tiles
      mbar_init(&q_empty[i], 1);
      mbar_init(&raw_full[i], 2);   // the box, and the unit's multipliers in sC
    }
    for (int i = 0; i < 2; ++i) {
      mbar_init(&e_full[i], kPairConsumers);
      mbar_init(&sel_done[i], 1);
      mbar_init(&acc_full[i], 1);
      mbar_init(&acc_empty[i], kPairConsumers);
    }
    for (int i = 0; i < kPairPieces; ++i) {
      mbar_init(&full[i], 1);
      mbar_init(&empty[i], 1);
    }
    mbar_init(&drain_bar, 1);
    fence_barrier_init();
  }
  if (warp == 4 * kPairGroups + 1) {
    tmem_alloc(&tmem_base_s, 512);
    tmem_relinquish();
  }
  tc_fence_before();
  __syncthreads();
  tc_fence_after();
  const uint32_t tmem = tmem_base_s;
  pdl_trigger();
  pdl_wait();
  // chunks of a unit: those of its last tile (the later tile of a pair has the larger candidate range)
  auto unit_chunks = [](const PairInfo& pi) { return (pi.sg[pi.nt - 1].J_hi + 128) >> 7; };

  if (warp == 4 * kPairGroups + 2) {
    // ---------------- set-up: unit k of this CTA is number blockIdx.x + k * gridDim.x of the planner's table
    // (heaviest first; a static round-robin, no atomic on the critical path).  Query tiles by TMA, one box per 64-element
    // half (FP8: one, see kQLeadRows); rows of a short last tile get whatever follows and are not used.
    const uint64_t pol = l2_policy_evict_first();
    bool live = true;   // no wait of this lane for a buffer has run out; after one it requests nothing more
    for (int k = 0;; ++k) {
      const int slot = k % kPairInfoSlots, qb = k % kPairQBufs;
      if (k >= kPairInfoSlots) mbar_wait(&info_empty[slot], ((k / kPairInfoSlots) - 1) & 1, ctx, 111);
      const int u = (int)blockIdx.x + k * (int)gridDim.x;
      bool valid = u < nunits && !*ctx.abort;   // after a wait has run out no further unit is started
      valid = __shfl_sync(0xffffffffu, valid, 0);
      if (lane == 0) {
        PairInfo& pi = info[slot];
        pi.valid = valid;
        if (valid) {
          const int2 un = units[u];
          pi.sg[0] = segs[un.x];
          pi.nt = un.y >= 0 ? 2 : 1;
          if (un.y >= 0) pi.sg[1] = segs[un.y];
        }
        __threadfence_block();
        mbar_arrive(&info_full[slot]);
      }
      __syncwarp();
      if (!valid) break;
      if (k >= kPairQBufs) live &= mbar_wait(&q_empty[qb], ((k / kPairQBufs) - 1) & 1, ctx, 112);
      const PairInfo& pi = info[slot];
      const SegInfo& sg = pi.sg[0];
      const int tok0 = sg.r0 / P.group, lead = sg.r0 - tok0 * P.group, nt = pi.nt;
      uint8_t* buf = sQ + qb * kPairQBytes;
      const CUtensorMap* mp = nt > 1 ? &map_q2 : &map_q;
      const uint32_t rows = (uint32_t)(P.group * (nt > 1 ? P.q_box2_tok : P.q_box_tok));
      if constexpr (FP8) {
        if (lane == 0 && live) {
          mbar_arrive_expect_tx(&raw_full[qb], rows * 128u);
          tma_load_3d_hint(buf + kPairQHalf - lead * 128, mp, &raw_full[qb], 0, sg.h * P.group, sg.q_tok0 + tok0, pol);
        }
        for (int j = lane; j < nt * kTileRows; j += 32)   // (adjacent tiles: row j of the pair is packed row r0 + j)
          sC[slot][j] = P.scale_log2 * q_scale[sg.h * P.group + (sg.r0 + j) % P.group];
        __syncwarp();
        if (lane == 0 && live) mbar_arrive(&raw_full[qb]);
      } else if (lane == 0 && live) {
        mbar_arrive_expect_tx(&q_full[qb], rows * 256u);
        tma_load_3d_hint(buf - lead * 128, mp, &q_full[qb], 0, sg.h * P.group, sg.q_tok0 + tok0, pol);
        tma_load_3d_hint(buf + kPairQHalf - lead * 128, mp, &q_full[qb], 64, sg.h * P.group, sg.q_tok0 + tok0, pol);
      }
      __syncwarp();
    }
  } else if (warp == 4 * kPairGroups + 3) {
    // ---------------- selection: threshold, forced blocks, ordered compaction of the tiles of unit `it` ----------------
    for (int it = 0;; ++it) {
      const int slot = it % kPairInfoSlots, eb = it & 1;
      const PairInfo& pi = info[slot];
      if (!ready_warp(&info_full[slot], (it / kPairInfoSlots) & 1, ctx, 151, &pi.valid)) break;
      mbar_wait(&e_full[eb], (it >> 1) & 1, ctx, 152);
      for (int tt = 0; tt < pi.nt; ++tt) {
        const SegInfo sg = pi.sg[tt];
        const int ncand = sg.J_hi + 1;
        const float* e = sE + (ncand > kMaxBlocks / 2 ? 0 : eb * (kMaxBlocks / 2) + tt * kPairMaxCand);
        float maxE = red[eb][tt][0];
#pragma unroll
        for (int i = 1; i < 4 * kPairGroups; ++i) maxE = fmaxf(maxE, red[eb][tt][i]);
        // J selected  <=>  E_J >= alpha max E  <=>  e_J >= log2(alpha) + max e   (alpha <= 0 selects everything)
        const float thr = P.alpha > 0.f ? maxE + log2f(P.alpha) : -INFINITY;
        const int win_lo = sg.J_lo - P.window_blocks;
        int pos = 0;
        for (int J0 = 0; J0 < ncand; J0 += 32) {
          const int J = J0 + lane;
          const bool keep = J < ncand && (e[J] >= thr || J < P.sink_blocks || J >= win_lo);
          const unsigned bal = __ballot_sync(0xffffffffu, keep);
          if (keep) blk_idx[sg.off + pos + __popc(bal & ((1u << lane) - 1u))] = J;
          pos += __popc(bal);
        }
        __syncwarp();
        if (lane == 0) {
          seg_count[sg.seg] = pos;
          seg_offset[sg.seg] = sg.off;
          if (sg.seg == P.nseg - 1) seg_offset[P.nseg] = sg.off + ncand;
        }
      }
      __syncwarp();
      if (lane == 0) {
        mbar_arrive(&sel_done[eb]);
        mbar_arrive(&info_empty[slot]);
      }
    }
  } else if (warp == 4 * kPairGroups) {
    // ---------------- producer: kbar pieces of every 128-block chunk (hi then lo, each in its two halves of d) ----------------
    if (lane == 0) {
      tma_prefetch_desc(&map_khi);
      tma_prefetch_desc(&map_klo);
      const uint64_t keep = l2_policy_evict_last();
      uint32_t pc = 0;
      auto produce = [&]() {
        for (int it = 0;; ++it) {
          const int slot = it % kPairInfoSlots;
          const PairInfo& pi = info[slot];
          if (!mbar_wait(&info_full[slot], (it / kPairInfoSlots) & 1, ctx, 121) || !pi.valid) break;
          const int h = pi.sg[0].h, blk_off = pi.sg[0].blk_off;
          const int nchunks = unit_chunks(pi);
          for (int c = 0; c < nchunks; ++c) {
  #pragma unroll
            for (int p = 0; p < 4; ++p, ++pc) {
              const int s = pc % kPairPieces;
              if (pc >= kPairPieces && !mbar_wait(&empty[s], ((pc / kPairPieces) - 1) & 1, ctx, 122)) return;   // nothing more after an abort
              mbar_arrive_expect_tx(&full[s], kPairPieceBytes);
              tma_load_3d_hint(sStage + s * kPairPieceBytes, p < 2 ? &map_khi : &map_klo, &full[s], (p & 1) * 64, h,
                               blk_off + c * 128, keep);
            }
          }
          mbar_arrive(&info_empty[slot]);
        }
      };
      produce();
    }
  } else if (warp == 4 * kPairGroups + 1) {
    // ---------------- UMMA issuer: acc[chunk & 1] = kbar_hi Q^T + kbar_lo Q^T over the unit's one or two tiles ----------------
    // the whole warp walks the loop, one elected lane issues (see the attention kernel's issuer)
    const bool leader = elect_one();
    constexpr int kFmt = FP8 ? 0 : 1;             // F16 / BF16 operands
    uint32_t pc = 0, ac0 = 0, ac1 = 0, gc0 = 0;   // gc0: chunks of all earlier units
    for (int it = 0;; ++it) {
      const int slot = it % kPairInfoSlots, qb = it % kPairQBufs;
      const PairInfo& pi = info[slot];
      if (!ready_warp(&info_full[slot], (it / kPairInfoSlots) & 1, ctx, 131, &pi.valid)) break;
      const int nchunks = unit_chunks(pi);
      const uint32_t idesc = make_idesc(128, 128 * pi.nt, kFmt, kFmt, 0, 0);
      mbar_wait(&q_full[qb], (it / kPairQBufs) & 1, ctx, 132);
      const uint64_t q_desc = make_smem_desc_sw128(smem_u32(sQ + qb * kPairQBytes), 16, 1024);
      for (int c = 0; c < nchunks; ++c) {
        const int a = (gc0 + c) & 1;
        uint32_t& ac = a ? ac1 : ac0;
        if (ac >= 1) mbar_wait(&acc_empty[a], (ac - 1) & 1, ctx, 133);
        ++ac;
#pragma unroll
        for (int p = 0; p < 4; ++p, ++pc) {
          const int s = pc % kPairPieces;
          const bool ready = mbar_wait(&full[s], (pc / kPairPieces) & 1, ctx, 134);
          tc_fence_after();
          const uint64_t a_desc = make_smem_desc_sw128(smem_u32(sStage + s * kPairPieceBytes), 16, 1024);
          if (leader && ready) {
#pragma unroll
            for (int ks = 0; ks < 4; ++ks)
              umma_f16_ss(tmem + a * 256, a_desc + ks * 2, q_desc + ((p & 1) * (kPairQHalf >> 4) + ks * 2), idesc, (p | ks) != 0);
            umma_commit(&empty[s]);
            if (p == 3) umma_commit(&acc_full[a]);
          }
        }
      }
      __syncwarp();   // no lane reads the descriptor any more
      if (leader) {
        umma_commit(&q_empty[qb]);
        mbar_arrive(&info_empty[slot]);
      }
      gc0 += nchunks;
    }
  } else {
    // ---------------- consumers: per pooled key and tile, maximum and exponential sum over the tile's rows ----------------
    const int wg = warp >> 2;
    const int key = (warp & 3) * 32 + lane;  // TMEM lane = pooled key within the chunk
    const uint32_t lane_base = tmem + ((uint32_t)((warp & 3) * 32) << 16);
    const float cs = P.scale_log2;
    uint32_t gc0 = 0;  // chunks of all earlier units
    int turn = 0;      // warpgroup whose turn the next item (chunk, tile) is
    bool prev_big = false;
    // FP8: the tiles of unit k from e4m3 to F16, for the MMAs.  Done one unit ahead, when the unit's raw box has had the time
    // of a unit's last chunk to land.
    auto widen_unit = [&](int k) {
      const PairInfo& pk = info[k % kPairInfoSlots];
      const int qb = k % kPairQBufs;
      if (!ready_warp(&info_full[k % kPairInfoSlots], (k / kPairInfoSlots) & 1, ctx, 145, &pk.valid)) return;
      mbar_wait(&raw_full[qb], (k / kPairQBufs) & 1, ctx, 114);
      uint8_t* const buf = sQ + qb * kPairQBytes;
      widen_pair_in_place(buf, buf + kPairQHalf, pk.nt * kTileRows, warp, lane);
      fence_proxy_async();
      __syncwarp();
      if (lane == 0) mbar_arrive(&q_full[qb]);
    };
    if constexpr (FP8) widen_unit(0);
    for (int it = 0;; ++it) {
      const int slot = it % kPairInfoSlots;
      const PairInfo& pi = info[slot];
      if (!ready_warp(&info_full[slot], (it / kPairInfoSlots) & 1, ctx, 141, &pi.valid)) break;
      if constexpr (FP8) widen_unit(it + 1);
      const int nt = pi.nt;
      const int nchunks = unit_chunks(pi);
      const int ncand0 = pi.sg[0].J_hi + 1, ncand1 = nt > 1 ? pi.sg[1].J_hi + 1 : 0;
      const int nrows0 = pi.sg[0].nrows, nrows1 = nt > 1 ? pi.sg[1].nrows : 0;
      // per candidate: log2 of its energy, e_J = m_J + log2(S_J)  (Eq. 1-2 / Eq. 20 in the log domain: the common
      // factor 2^-M of Eq. 20 cancels in the comparison with alpha * max)
      float lmax0 = -INFINITY, lmax1 = -INFINITY;
      const int eb = it & 1;
      const bool big = ncand0 > kMaxBlocks / 2;    // a single tile that takes the whole energy buffer
      float* e0 = sE + (big ? 0 : eb * (kMaxBlocks / 2));
      float* e1 = e0 + kPairMaxCand;
      // the part of the energy buffer this unit writes must have been read by the selection of unit it-2, and a unit
      // that takes (or follows one that took) the whole buffer also waits for unit it-1
      if (it >= 2) mbar_wait(&sel_done[eb], ((it >> 1) - 1) & 1, ctx, 143);
      if (it >= 1 && (big || prev_big)) mbar_wait(&sel_done[eb ^ 1], ((it - 1) >> 1) & 1, ctx, 144);
      prev_big = big;
      // Accumulators alternate by a chunk count that runs across units, items by a turn that does.  Every warpgroup waits for
      // every chunk and hands its accumulator back, also where it has no item of the chunk: a warpgroup that were passed by
      // two chunks of one accumulator could not tell the barrier's phases apart.
      for (int c = 0; c < nchunks; ++c) {
        const uint32_t n = gc0 + (uint32_t)c;
        const int a = (int)(n & 1u);
        mbar_wait(&acc_full[a], (n >> 1) & 1, ctx, 142);
        int tt = wg - turn;                        // this warpgroup's tile of the chunk, if below nt
        if (tt < 0) tt += kPairGroups;
        turn = turn + nt >= kPairGroups ? turn + nt - kPairGroups : turn + nt;
        if (tt >= nt) {
          mbar_arrive(&acc_empty[a]);
          continue;
        }
        tc_fence_after();
        const int J = c * 128 + key;
        const int nrows = tt ? nrows1 : nrows0;
        const uint32_t lane_addr = lane_base + a * 256 + tt * 128;
        const float* mult = &sC[FP8 ? slot : 0][FP8 ? tt * kTileRows : 0];
        const float e = nrows == kTileRows ? score_cols<FP8, NP, false>(lane_addr, cs, mult, kTileRows, &acc_empty[a])
                                           : score_cols<FP8, NP, true>(lane_addr, cs, mult, nrows, &acc_empty[a]);
        if (J < (tt ? ncand1 : ncand0)) {
          (tt ? e1 : e0)[J] = e;
          if (tt) lmax1 = fmaxf(lmax1, e);
          else lmax0 = fmaxf(lmax0, e);
        }
      }
#pragma unroll
      for (int o = 16; o > 0; o >>= 1) {
        lmax0 = fmaxf(lmax0, __shfl_xor_sync(0xffffffffu, lmax0, o));
        lmax1 = fmaxf(lmax1, __shfl_xor_sync(0xffffffffu, lmax1, o));
      }
      // hand the unit to the selection warp and go on
      if (lane == 0) {
        red[eb][0][warp] = lmax0;
        red[eb][1][warp] = lmax1;
      }
      __syncwarp();
      mbar_arrive(&e_full[eb]);
      mbar_arrive(&info_empty[slot]);
      gc0 += (uint32_t)nchunks;
    }
  }
  leave_cta(ctx, &drain_bar, warp == 4 * kPairGroups + 1);
  if (warp == 4 * kPairGroups + 1) tmem_dealloc(tmem, 512);
}

}  // namespace fp2
