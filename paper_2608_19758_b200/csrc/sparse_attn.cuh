// Block-sparse causal flash attention with mean correction (Eq. 4, Eq. 6; Algorithm 1 lines 6-11),
// persistent, warp-specialised, tcgen05 / TMEM / TMA.  The same kernel runs the dense path (implicit list
// 0..J_hi, no correction).
//
// CTAs loop over work units (sequence, KV head, packed query tile) taken from a work order (long ones of all heads
// first, then KV-head-major, see order_scatter_kernel) through a global counter.  For a unit with selected list idx[0..T) the iteration sequence
// is the list traversed backwards (Eq. 17) followed by the non-empty correction chunks: a correction chunk
// stages 128 consecutive pooled (kbar, vbar) rows exactly like a KV block, its logits are shifted by log2(128)
// (every corrected block is full) and masked by todo = fully-visible & ~selected.
//
// TWO small CTAs per SM.  Per 128x128 block the tensor pipe (two GEMMs) and the MUFU pipe (16384
// exponentials) are each busy 1024 cycles, and a softmax step has several hundred cycles of latency around its
// exponentials (TMEM load, row maximum, TMEM store, barrier hand-overs).  Two warpgroups that share one tile must
// exchange row maxima and so move in lockstep: both are in their latency phase at the same time and the MUFU
// pipe idles (that layout, one CTA of 12 warps per SM, measured 42-48 % tensor-pipe activity on the dense
// path; this one 59 %).  Here every CTA has ONE softmax warpgroup that owns whole rows (thread = row, 128 logits
// in registers), nothing crosses between the two CTAs of an SM, and they drift out of phase by themselves: while
// one CTA's warps stream exponentials the other's wait for the tensor pipe, load logits or hand over P.
//
// One CTA: 256 threads, 96 KB of tile memory (Q, one K stage, one V stage), 256 TMEM columns:
//   S [0,128)  logits of the iteration; P (16-bit pairs) overwrites its first 64 columns in place
//   O [128,256)
// Everything is single-buffered: S = Q K^T of iteration i+1 is issued behind O += P V of iteration i (which
// reads P out of the S columns), the K tile of i+1 is requested when S = Q K^T (i) has completed and the V tile
// when O += P V (i) has.  The other CTA of the SM fills the bubbles this leaves.  P is handed to the issuer in
// kPParts column slices (see PSlices), so O += P V runs its first k-steps under the remaining exponentials.
//
// Roles: warps 0..3 softmax + epilogue; warp 4 TMA producer (Eq. 22); warp 5 UMMA issuer (and TMEM owner);
// warps 6, 7 unit set-up (fetch the next unit, validate its list, build the correction masks, stage Q).
//
// FP8 inputs (Eq. 15; template parameter FP8): S = Q K^T runs as a kind::f8f6f4 MMA straight on the raw e4m3
// tiles (Q and K both K-major, 128-byte rows, as cp.async / TMA write them), at twice the BF16 rate.  The
// probabilities stay 16-bit -- a single e4m3 probability tile costs ~0.06 max-abs output error by itself -- so
// O += P V is a kind::f16 MMA on F16 operands: P packed as F16, V an F16 copy made for the call in the workspace
// (attn_prepare_kernel; one contiguous tile per block; map_v is its map).  Short calls and callers without a workspace
// (template parameter WIDEN) have no such copy: there the softmax warpgroup widens (exactly) the raw e4m3 tile into the F16
// V stage at the top of the iteration.
// The per-head scales never touch the operands: q_scale * k_scale multiplies the logits of a row, v_scale multiplies the
// output.  Correction chunks: the pooled keys come as an e4m3 hi + lo pair in raw units (two accumulating MMA groups, ~8
// mantissa bits together), the pooled values as F16.  Tile memory: Q 16 KB, K 32 KB (one raw tile, or hi | lo of a
// chunk), F16 V 32 KB (raw V 16 KB).
// 16384 tokens dense, 28 heads on 4 KV heads: 1723 us widening per iteration, 1456 us with the copy (its 11 us included).
#pragma once
#include <cuda_bf16.h>
#include "common.cuh"
#include "ptx.cuh"
#include "score_select.cuh"  // load_q_tile_async
#include "split_kv.cuh"

namespace fp2 {

constexpr int kTileBytes = 32768;   // one 128 x 128 tile of 16-bit elements
constexpr int kRawBytes = 16384;    // one 128 x 128 tile of FP8 elements as TMA delivers it

struct TileInfo {
  SegInfo sg;
  int32_t valid;     // 0: no more work
  int32_t T;         // exact iterations (listed blocks)
  int32_t nchunk;    // non-empty correction chunks
  int32_t ndiag;     // listed blocks J >= J_lo: the first ndiag iterations (the list is traversed backwards)
  int32_t dense;
  int32_t it_begin, it_end;   // this unit's part of the iteration sequence [0, T + nchunk) (Eq. 18); all of it unless split
  int32_t parts;              // parts the segment is split into (1: the unit writes the final output)
  int32_t slot;               // partial-result slot of this unit when parts > 1
  int32_t chunk_id[kMaxChunks];
  uint32_t todo[kMaxChunks][4];
};

struct AttnArgs {
  const uint8_t* q;
  const int32_t* page_table;
  const SegInfo* segs;
  const int32_t* order;      // work order
  const int32_t* seg_count;  // NULL => dense
  const int32_t* blk_idx;
  const float* q_scale;
  const float* k_scale;
  const float* v_scale;
  __nv_bfloat16* out;
  float* lse;
  int* work_counter;
  int* status;
  // KV splitting (Eq. 18).  unit_split == NULL: one unit per segment, `order` lists the segments.  Otherwise
  // `order` lists the segment of every unit, unit_split its part (see pack_split), *n_units their number, and a
  // unit of a split segment leaves (O, m, l) unnormalised in part_o [slot][128][128] / part_ml [slot][128].
  const int32_t* unit_split;
  const int32_t* n_units;
  float* part_o;
  float2* part_ml;
#ifdef FP2_PROFILE
  long long* prof;   // [grid][16] cycle counters of the softmax warpgroup (development builds only)
#endif
};

#ifdef FP2_PROFILE
#define PF_BEGIN() pf_a = clock64()
#define PF_END(k) (pf_b = clock64(), pf[k] += pf_b - pf_a, pf_a = pf_b)
#else
#define PF_BEGIN()
#define PF_END(k)
#endif

// P is handed to the issuer in column slices.  Each hand-over stalls the warp for its TMEM stores, and what follows the last one
// (the slice's MMAs, then S = Q K^T) is what the warp waits for; so: a short first slice to get O += P V going, a long middle
// one, a short last one.  In k-steps (of eight), whole calls in us, in turn: 4 x 2 / 4 + 4 / 2 + 5 + 1 / 2 + 4 + 2: 32768 tokens
// dense BF16 8090 / 8050 / 7786 / 7615, 32768 tokens 1794 / 1775 / 1739 / 1728, 131072 tokens 10980 / 10923 / 10722 / 10611, 16
// sequences within 1 %; FP8 16384 tokens dense 1509 / 1506 / 1456 / 1518, 131072 tokens 7872 / 7882 / 7715 / 7898, 8191 tokens
// 200.6 / 200.2 / 196.2 / 199.7, 16 sequences within 1 %.  16 columns a store, except FP8, whose middle slice ends inside 16.
constexpr int kPParts = 3;
template <bool FP8>
struct PSlices {
  static constexpr int kStore = FP8 ? 8 : 16;   // packed registers (= P columns) per TMEM store
  // k-steps (16 probabilities of a row, 8 columns) that are there once slice h is
  __host__ __device__ static constexpr int end(int h) { return h == 0 ? 2 : h == 1 ? (FP8 ? 7 : 6) : 8; }
  // slice that is complete after this many k-steps, -1: none
  __host__ __device__ static constexpr int complete(int steps) {
    for (int h = 0; h < kPParts; ++h)
      if (end(h) == steps) return h;
    return -1;
  }
};

template <bool FP8>
struct AttnCfg {
  static constexpr int kThreads = 256;
  static constexpr int kCtasPerSm = 2;
  static constexpr int kBiasBytes = 4096;                    // one 128 x 32 e5m2 operand without swizzle
  // query tile: per 128 bytes of a row (two halves BF16, one FP8) 128 rows and the overhang of the box (see kQLeadRows)
  static constexpr int kQHalf = 16384 + kQTailRows * 128;
  static constexpr int kOffK = kQLeadRows * 128 + (FP8 ? 1 : 2) * kQHalf;
  static constexpr int kOffHot = kOffK + 2 * kTileBytes + (FP8 ? kRawBytes : 0);
  static constexpr int kSmemBytes = 1024 + kOffHot + 2 * kBiasBytes;   // 98 to 101 KB of tiles + the mask operands
  // Registers: two CTAs share the file, 128 per thread at launch; setmaxnreg moves them from the service warps
  // to the softmax warps.  The move waits without bound for registers the CTA does not own, so the sum is
  // checked here and the compiled register count is checked on the host before the first launch.
  static constexpr int kRegsBase = 128;
  static constexpr int kRegsService = 56;
  static constexpr int kRegsSoftmax = 200;
  static constexpr int kRegsAfterMove = (kThreads - 128) * kRegsService + 128 * kRegsSoftmax;
  static_assert(kRegsAfterMove <= kThreads * kRegsBase, "register budget: setmaxnreg.inc would wait forever");
  static_assert(kThreads * kRegsBase * kCtasPerSm <= 65536, "two CTAs must fit the register file");
};

// Masked iterations (diagonal blocks, correction chunks -- the minority): overwrite the hidden logits of this
// thread's row with -inf in TMEM, so that the softmax step itself carries no mask logic.  Column j stays
// visible iff j <= tok_lim and bit j of the 128-bit mask (32 bits per word) is set.  Not inlined: it is off the
// common path and four times 32 unrolled selects are a lot of code.
__device__ __noinline__ void mask_row(uint32_t s_addr, int tok_lim, uint32_t cm0, uint32_t cm1, uint32_t cm2,
                                      uint32_t cm3) {
#pragma unroll 1
  for (int k = 0; k < 4; ++k) {
    const uint32_t cmk = k == 0 ? cm0 : k == 1 ? cm1 : k == 2 ? cm2 : cm3;
    const bool all_vis = (k * 32 + 31 <= tok_lim) && (cmk == 0xffffffffu);
    if (__all_sync(0xffffffffu, all_vis)) continue;   // TMEM accesses are warp-wide: decide per warp
    uint32_t rr[32];
    tmem_ld32(s_addr + k * 32, rr);
    tmem_wait_ld();
#pragma unroll
    for (int j = 0; j < 32; ++j) {
      const bool vis = (k * 32 + j <= tok_lim) && ((cmk >> j) & 1u);
      rr[j] = vis ? rr[j] : 0xff800000u;  // -inf
    }
    tmem_st32(s_addr + k * 32, rr);
  }
  tmem_wait_st();
}

// The thread's whole logit row (raw, unscaled) into registers, and its maximum: all four TMEM loads in flight,
// chains of three-input maxima.
__device__ __forceinline__ float row_load_max(uint32_t s_addr, uint32_t (&x)[128]) {
#pragma unroll
  for (int k = 0; k < 4; ++k) tmem_ld32(s_addr + k * 32, reinterpret_cast<uint32_t(&)[32]>(x[k * 32]));
  tmem_wait_ld();
  float mx8[16];
#pragma unroll
  for (int c = 0; c < 16; ++c) {
    const float* v = reinterpret_cast<const float*>(&x[c * 8]);
    mx8[c] = fmaxf(max3(max3(v[0], v[1], v[2]), v[3], v[4]), max3(v[5], v[6], v[7]));
  }
#pragma unroll
  for (int c = 0; c < 5; ++c) mx8[c] = max3(mx8[3 * c], mx8[3 * c + 1], mx8[3 * c + 2]);
  return fmaxf(max3(mx8[0], mx8[1], mx8[2]), max3(mx8[3], mx8[4], mx8[15]));
}

// p = 2^(x * cs + neg_m) for the 128 logits in registers, written as BF16 (F16) pairs to the 64 columns at p_addr.
// Scaling and row sum use packed fp32x2 instructions.  The thread arrives on part_ready as the slices (but the last) are
// complete.  Returns the row sum.
template <bool F16>
__device__ __forceinline__ float row_exp(const uint32_t (&x)[128], uint32_t p_addr, float cs, float neg_m,
                                         uint64_t* part_ready) {
  const uint64_t cs2 = f2_pack(cs, cs), nm2 = f2_pack(neg_m, neg_m);
  uint64_t sum2[4] = {0ull, 0ull, 0ull, 0ull};   // four independent (lo, hi) accumulators, +0.0f bit patterns
  using Slices = PSlices<F16>;
  constexpr int W = Slices::kStore;
#pragma unroll
  for (int k = 0; k < 64 / W; ++k) {
    uint32_t pk[W];
#pragma unroll
    for (int j = 0; j < W; ++j) {
      const int c = k * 2 * W + 2 * j;
      const uint64_t x2 = f2_fma(f2_pack(__uint_as_float(x[c]), __uint_as_float(x[c + 1])), cs2, nm2);
      float x0, x1;
      f2_unpack(x2, x0, x1);
      const float p0 = ex2(x0), p1 = ex2(x1);
      sum2[j & 3] = f2_add(sum2[j & 3], f2_pack(p0, p1));
      pk[j] = F16 ? pack_f16x2(p0, p1) : pack_bf16x2(p0, p1);
    }
    tmem_st_cols(p_addr + k * W, pk);
    const int slice = Slices::complete((k + 1) * W / 8);
    if (slice >= 0 && slice + 1 < kPParts) {   // O += P V may run the slice's k-steps
      tmem_wait_st();
      tc_fence_before();
      mbar_arrive(&part_ready[slice]);
    }
  }
  float a0, a1;
  f2_unpack(f2_add(f2_add(sum2[0], sum2[1]), f2_add(sum2[2], sum2[3])), a0, a1);
  return a0 + a1;
}

// map_kbar / map_kbar_lo: pooled keys of the correction chunks -- BF16: one BF16 array (map_kbar_lo unused);
// FP8: the e4m3 hi and lo arrays.  map_vbar: pooled values, 16-bit.  map_q: packed query tiles (DevParams::q_box).
template <bool FP8, bool WIDEN>
__global__ void __launch_bounds__(AttnCfg<FP8>::kThreads, AttnCfg<FP8>::kCtasPerSm)
sparse_attn_kernel(const __grid_constant__ CUtensorMap map_k, const __grid_constant__ CUtensorMap map_v,
                    const __grid_constant__ CUtensorMap map_kbar, const __grid_constant__ CUtensorMap map_kbar_lo,
                    const __grid_constant__ CUtensorMap map_vbar, const __grid_constant__ CUtensorMap map_q,
                    AttnArgs A, DevParams P) {
  constexpr int kSetupThreads = 64;
  extern __shared__ uint8_t smem_raw[];
  uint8_t* smem = reinterpret_cast<uint8_t*>((reinterpret_cast<uintptr_t>(smem_raw) + 1023) & ~uintptr_t(1023));
  uint8_t* sQ = smem + kQLeadRows * 128;               // 32 KB (BF16) / 16 KB (raw e4m3) and padding
  uint8_t* sK = smem + AttnCfg<FP8>::kOffK;            // 32 KB
  uint8_t* sV = sK + kTileBytes;                       // 32 KB, 16-bit
  uint8_t* sVraw = sV + kTileBytes;                    // WIDEN only: 16 KB raw e4m3 V tile
  (void)sVraw;
  // Masks enter the logits through the tensor core: one more k-step S += hot . bias^T (kind::f8f6f4, e5m2 x e5m2,
  // K = 32), which costs 64 cycles of the tensor pipe instead of a TMEM round trip of the softmax warpgroup.
  //   sHot [128 rows x 32]: row i holds 57344 (the largest e5m2) in column c(i) and zeros elsewhere, c(i) = the
  //     row's position minus the tile's first position (Eq. 13: floor((r0 + i) / g) - floor(r0 / g)); written by the
  //     set-up warps with the query tile.  Group sizes with more than 32 positions per tile (g < 4) use i mod 32.
  //   sBias [128 columns x 32], written by the producer warp per masked iteration:
  //     diagonal block: bias[j][c] = -57344 where column j is hidden from position c (j > t0 + c), else 0;
  //     correction chunk: bias[j][c] = -57344 for every c where block j is not to be corrected (selected, or past
  //       the fully visible range), else 0 -- the todo mask is the same for all rows.
  // A hidden logit thus carries -3.3e9 (raw units), which the exponential turns into an exact zero.
  // Both operands are K-major without swizzle: 8-row x 16-byte core matrices, row r at (r / 8) * 256 + (r % 8) * 16,
  // bytes 16..31 of the row 128 bytes further.
  uint8_t* sHot = smem + AttnCfg<FP8>::kOffHot;
  uint8_t* sBias = sHot + AttnCfg<FP8>::kBiasBytes;

  __shared__ TileInfo info[2];
  __shared__ uint32_t sel_bits[kMaxBlocks / 32];
  __shared__ uint64_t info_full[2], info_empty[2], q_full, q_empty;
  // Every barrier below completes exactly once per iteration; with G the iteration's index counted over the
  // whole kernel, the phase that belongs to iteration G has parity G & 1.
  __shared__ uint64_t k_full, v_full;
  __shared__ uint64_t s_done;    // S = Q K^T (G) has completed: the logits are in TMEM, the K stage is free --
                                 // and, MMAs completing in issue order, O += P V (G-1) is in O
  __shared__ uint64_t pv_done[2];  // [G & 1], phase (G >> 1) & 1: O += P V (G) has completed -- the V stage is free,
                                   // O holds iteration G.  Two barriers so that a waiter may be two iterations
                                   // behind the issuer without mistaking one phase for another.
  __shared__ uint64_t vraw_full, vraw_empty;   // WIDEN: the raw V tile has landed / has been widened
  __shared__ uint64_t p_ready[kPParts];   // slice q (see PSlices) of P (G) is in TMEM
  __shared__ uint32_t tmem_base_s;
  __shared__ int abort_flag;
  __shared__ int ndiag_s, unit_s;
  __shared__ uint64_t drain_bar;   // teardown after an abort: every MMA issued by this CTA has completed

  const int tid = threadIdx.x, warp = tid >> 5, lane = tid & 31;
  WaitCtx ctx{A.status, &abort_flag};

  if (tid == 0) {
    abort_flag = 0;
    for (int i = 0; i < 2; ++i) {
      mbar_init(&info_full[i], 1);
      mbar_init(&info_empty[i], 2 + 128);   // producer, issuer, softmax threads
    }
    mbar_init(&q_full, kSetupThreads + (P.q_box ? 1 : 0));
    mbar_init(&vraw_full, 1);
    mbar_init(&vraw_empty, 4);   // one arrival per softmax warp
    mbar_init(&q_empty, 1);
    mbar_init(&k_full, 1);
    mbar_init(&v_full, WIDEN ? 4 : 1);   // WIDEN: the softmax warps', or the producer's for all of them
    mbar_init(&s_done, 1);
    mbar_init(&pv_done[0], 1);
    mbar_init(&pv_done[1], 1);
    mbar_init(&drain_bar, 1);
    for (int i = 0; i < kPParts; ++i) mbar_init(&p_ready[i], 128);
    fence_barrier_init();
  }
  // K / V stages start zeroed: rows of pages past the end of a sequence are never loaded, and whatever sits
  // there is multiplied by probabilities that are exactly zero, so it must be finite.
  for (int i = tid; i < (2 * kTileBytes + (FP8 ? kRawBytes : 0)) / 16; i += AttnCfg<FP8>::kThreads)
    reinterpret_cast<uint4*>(sK)[i] = make_uint4(0, 0, 0, 0);
  if (warp == 5) {
    tmem_alloc(&tmem_base_s, 256);
    tmem_relinquish();
  }
  fence_proxy_async();
  tc_fence_before();
  __syncthreads();
  tc_fence_after();
  const uint32_t tmem = tmem_base_s;
  if (tid == 0) {   // (kernel parameters: no need to wait for the kernel before)
    tma_prefetch_desc(&map_k);
    tma_prefetch_desc(&map_v);
    tma_prefetch_desc(&map_kbar);
    tma_prefetch_desc(&map_vbar);
    if (P.q_box) tma_prefetch_desc(&map_q);
  }
  pdl_trigger();
  pdl_wait();
  const int g = P.group;

  // O += P V (G) has completed.  Safe for a waiter that is at most two iterations behind the issuer.
  auto wait_pv = [&](uint32_t G, int where) { return mbar_wait(&pv_done[G & 1], (G >> 1) & 1, ctx, where); };

  if (warp >= 6) {
    // =============================== unit set-up + Q staging ===============================
    // A chain of dependent global loads (work counter -> order -> segment and count -> list -> page table), which at the start
    // of a call nothing hides: both warps load what they need themselves instead of passing it on, the page-table entries of
    // the list go to the L1 for the producer, the first unit is the CTA's own number, and its query tile is requested as soon
    // as the segment is known.  2048 tokens: logits of the first block after 8000 cycles of the kernel (9100 before).  Whole calls,
    // together with the issuer's look-ahead: 2048 tokens 35.8 -> 34.3 us, 2370 tokens 43.4 -> 41.2; long ones within 1 %.
    setmaxnreg_dec<AttnCfg<FP8>::kRegsService>();
    const int t64 = tid - 32 * 6;
    const bool corr = P.use_correction != 0;
    auto issue_q = [&](const SegInfo& sg) {
      // one TMA box per 128 bytes of a row (see kQLeadRows), landing in the swizzled layout the MMA reads.  Rows past the
      // end of a short last tile get whatever follows; nothing reads them.
      const uint64_t pol = l2_policy_evict_first();
      const int tok0 = sg.r0 / g;
      uint8_t* dst = sQ - (sg.r0 - tok0 * g) * 128;
      const uint32_t bytes = (uint32_t)(g * P.q_box_tok) * 128u;
      mbar_arrive_expect_tx(&q_full, FP8 ? bytes : 2 * bytes);
      tma_load_3d_hint(dst, &map_q, &q_full, 0, sg.h * g, sg.q_tok0 + tok0, pol);
      if constexpr (!FP8)
        tma_load_3d_hint(dst + AttnCfg<FP8>::kQHalf, &map_q, &q_full, 64, sg.h * g, sg.q_tok0 + tok0, pol);
    };
    if (t64 < 32)
      for (int w = t64; w < kMaxBlocks / 32; w += 32) sel_bits[w] = 0u;
    if (t64 == 0) ndiag_s = 0;
    const int n_units = A.unit_split ? *A.n_units : P.nseg;
    // Both warps run through the same named barriers whatever a wait gives: they leave by unit_s alone, which one thread sets.
    for (int it = 0;; ++it) {
      const int slot = it & 1;
      if (it >= 2) mbar_wait(&info_empty[slot], ((it >> 1) - 1) & 1, ctx, 201);
      TileInfo& ti = info[slot];
      if (t64 == 0) {
        const int w = it == 0 ? (int)blockIdx.x : (int)gridDim.x + atomicAdd(A.work_counter, 1);
        // after a wait has run out somewhere in this CTA no further unit is started: the terminating descriptor
        // makes every role leave its loop the ordinary way
        unit_s = w < n_units && !*ctx.abort ? w : -1;
      }
      named_bar_sync(2, kSetupThreads);   // (also: sel_bits and ndiag_s are clear)
      const int w = unit_s;
      if (w < 0) {
        if (t64 == 0) {
          ti.valid = 0;
          mbar_arrive(&info_full[slot]);
        }
        break;
      }
      const int seg = A.order[w];
      const SegInfo sg = A.segs[seg];
      const bool dense = A.seg_count == nullptr;
      int T = dense ? sg.J_hi + 1 : A.seg_count[seg];
      if (T < 0 || T > sg.J_hi + 1) {  // malformed count: clamp so every loop stays bounded
        if (t64 == 0) atomicOr(A.status + ST_BAD_LIST, 1);
        T = max(0, min(T, sg.J_hi + 1));
      }
      if (it == 0 && P.q_box && t64 == 0) issue_q(sg);
      if (!dense) {
        const int32_t* list = A.blk_idx + sg.off;
        const int32_t* pt = A.page_table + (size_t)sg.b * P.max_pages_per_seq;
        bool bad = false;
        int nd = 0;
#pragma unroll 1
        for (int k = t64; k < T; k += kSetupThreads) {
          const int J = list[k];
          const bool in = J >= 0 && J <= sg.J_hi;
          if (!in || (k > 0 && list[k - 1] >= J)) bad = true;
          if (in) prefetch_l1(pt + J * P.pages_per_block);
          if (corr && in && J < sg.J_lo) atomicOr(&sel_bits[J >> 5], 1u << (J & 31));
          nd += J >= sg.J_lo;
        }
        if (bad) atomicOr(A.status + ST_BAD_LIST, 1);
        nd = __reduce_add_sync(0xffffffffu, nd);
        if ((t64 & 31) == 0 && nd) atomicAdd(&ndiag_s, nd);
      }
      named_bar_sync(2, kSetupThreads);
      if (t64 < 32) {
        int nchunk = 0;
        if (!dense && corr) {   // chunk c: the pooled blocks that are fully visible and not listed
          const int c = t64;
          bool some = false;
          if (c * 128 < sg.J_lo) {
#pragma unroll
            for (int w2 = 0; w2 < 4; ++w2) {
              const int first = c * 128 + w2 * 32;
              uint32_t validm = 0u;
              if (first + 32 <= sg.J_lo) validm = 0xffffffffu;
              else if (first < sg.J_lo) validm = (1u << (sg.J_lo - first)) - 1u;
              const uint32_t todo = (first < sg.J_lo ? ~sel_bits[first >> 5] : 0u) & validm;
              ti.todo[c][w2] = todo;
              sel_bits[first >> 5] = 0u;
              some |= todo != 0u;
            }
          }
          const unsigned bal = __ballot_sync(0xffffffffu, some);
          if (some) ti.chunk_id[__popc(bal & ((1u << c) - 1u))] = c;
          nchunk = __popc(bal);
        }
        if (t64 == 0) {
          const int32_t split = A.unit_split ? A.unit_split[w] : pack_split(0, 1, 0);
          const int parts = (split >> 8) & 0xff, u = split & 0xff, n = T + nchunk;
          ti.sg = sg;
          ti.valid = 1;
          ti.dense = dense;
          ti.T = T;
          ti.nchunk = nchunk;
          ti.ndiag = dense ? min(T, sg.J_hi - sg.J_lo + 1) : ndiag_s;
          ndiag_s = 0;
          ti.parts = parts;
          ti.slot = ((split >> 16) & 0xffff) + u;
          // Eq. 18: part u of U takes iterations [u ceil(n / U), min((u + 1) ceil(n / U), n))
          const int step = parts == 1 ? n : (n + parts - 1) / parts;
          ti.it_begin = min(u * step, n);
          ti.it_end = min((u + 1) * step, n);
        }
        __syncwarp();
        if (t64 == 0) mbar_arrive(&info_full[slot]);
      }
      // Q tile: wait until every S = Q K^T of the previous unit has completed, then overwrite
      if (it >= 1) {
        const bool free = mbar_wait(&q_empty, (it - 1) & 1, ctx, 202);
        if (P.q_box && t64 == 0 && free) issue_q(sg);
      }
      {   // sHot: rows 2 t64 and 2 t64 + 1
        const int rem = sg.r0 % g;
#pragma unroll
        for (int u = 0; u < 2; ++u) {
          const int row = 2 * t64 + u;
          const int c = P.diag_mma ? (rem + row) / g : (row & 31);
          uint32_t w8[8] = {0u, 0u, 0u, 0u, 0u, 0u, 0u, 0u};
#pragma unroll
          for (int k = 0; k < 8; ++k) w8[k] = (c >> 2) == k ? 0x7bu << ((c & 3) * 8) : 0u;   // e5m2 57344
          uint8_t* dst = sHot + (row >> 3) * 256 + (row & 7) * 16;
          *reinterpret_cast<uint4*>(dst) = make_uint4(w8[0], w8[1], w8[2], w8[3]);
          *reinterpret_cast<uint4*>(dst + 128) = make_uint4(w8[4], w8[5], w8[6], w8[7]);
        }
        fence_proxy_async();
      }
      if (P.q_box) {
        mbar_arrive(&q_full);   // (one arrival more than threads: the byte count's)
        continue;
      }
      if constexpr (FP8) {
        load_q_raw_async(sQ, A.q, sg, P, t64, kSetupThreads);
        cp_async_wait_all();
      }
      else load_q_tile_async<AttnCfg<FP8>::kQHalf>(sQ, A.q, sg, P, t64, kSetupThreads);
      fence_proxy_async();
      mbar_arrive(&q_full);
    }
  } else if (warp == 4) {
    // =============================== TMA producer ===============================
    setmaxnreg_dec<AttnCfg<FP8>::kRegsService>();
    uint32_t G = 0, rc = 0;
    (void)rc;
    const uint64_t keep = l2_policy_evict_last();   // K / V pages and pooled means: shared by many tiles
    const int ppb = P.pages_per_block, psz = P.page_size;
    bool live = true;   // no wait of this lane has run out; after one it requests nothing more (the stages may not be free)
    for (int it = 0;; ++it) {
      const int slot = it & 1;
      const TileInfo& ti = info[slot];
      if (!ready_warp(&info_full[slot], (it >> 1) & 1, ctx, 301, &ti.valid)) break;
      const SegInfo& sg = ti.sg;
      const int T = ti.T;
      const int32_t* list = A.blk_idx + sg.off;
      const int32_t* pt = A.page_table + (size_t)sg.b * P.max_pages_per_seq;
      // page id of this lane's page of exact iteration i (-1: past the end of the sequence, or not an exact
      // iteration).  Fetched one iteration ahead, behind the K tile's copies: list entry -> page-table entry are two dependent
      // global loads, and the first K tile of a unit should not wait for the second's.
      int J_fetched = 0;   // block id of the iteration fetch_pid was last asked for (warp-uniform)
      auto fetch_pid = [&](int i) -> int {
        if (i >= T) return -1;
        int J = ti.dense ? sg.J_hi - i : list[T - 1 - i];
        J = max(0, min(J, sg.J_hi));
        J_fetched = J;
        if (lane >= ppb) return -1;
        if (J * kBlock + lane * psz >= sg.Lk) return -1;
        int pid = pt[J * ppb + lane];
        if (pid < 0 || pid >= P.num_pages) {
          atomicOr(A.status + ST_BAD_LIST, 2);
          pid = -1;
        }
        return pid;
      };
      // hidden columns of a masked iteration -> sBias (see there); row j = lane * 4 + u gets 32 bytes of which those of the
      // positions it is hidden from, the first ones, are -57344 (e5m2 0xfb).  The S = Q K^T that last read sBias has completed
      // (wait 302).  As little code as that takes, for the instruction cache.
      auto bias_row = [&](int u, const uint32_t (&w)[8]) {
        const int j = lane * 4 + u;
        uint8_t* dst = sBias + (j >> 3) * 256 + (j & 7) * 16;
        *reinterpret_cast<uint4*>(dst) = make_uint4(w[0], w[1], w[2], w[3]);
        *reinterpret_cast<uint4*>(dst + 128) = make_uint4(w[4], w[5], w[6], w[7]);
      };
      // The K tile of an iteration and its mask.  BF16: the copies go out first and do not wait for the mask; the phase of k_full
      // completes only with the arrival behind it, whatever has landed by then.  FP8, whose tile is half as large: the mask first;
      // the other way round dense calls are slower.  Whole calls in us, in turn, mask first / copies first: 131072 tokens 10398 /
      // 10361, last 8192 of them 1313 / 1305, 32768 tokens dense 7584 / 7562, the last 512 of them 361.2 / 354.5, 16 sequences
      // 3455 / 3444, 24 short sequences 151.5 / 151.1; FP8 dense 16384 tokens 1440.1 / 1447.2, 1500 tokens 39.6 / 40.6, 8191 tokens
      // 170.7 / 172.5, 131072 tokens within 0.2 %.
      auto request_k = [&](uint32_t bytes, auto copies, auto mask) {
        if constexpr (!FP8) copies();
        mask();
        if (lane == 0 && live) mbar_arrive_expect_tx(&k_full, bytes);
        if constexpr (FP8) copies();
      };
      int pid_next = fetch_pid(ti.it_begin);
      for (int i = ti.it_begin; i < ti.it_end; ++i, ++G) {
        const int pid = pid_next;
        const int J_cur = J_fetched;
        if (G >= 1) live &= mbar_wait(&s_done, (G - 1) & 1, ctx, 302);   // K stage free
        if (i < T) {
          const int nvalid = __popc(__ballot_sync(0xffffffffu, pid >= 0));
          const uint32_t bytes = (uint32_t)nvalid * psz * (FP8 ? 128u : 256u);
          request_k(bytes, [&]() {
            if constexpr (FP8) __syncwarp();
            if (pid >= 0 && live) {   // (FP8: the raw e4m3 tile, which the MMA reads as it lands)
              tma_load_3d_hint(sK + lane * psz * 128, &map_k, &k_full, 0, sg.h, pid * psz, keep);
              if constexpr (!FP8) tma_load_3d_hint(sK + 16384 + lane * psz * 128, &map_k, &k_full, 64, sg.h, pid * psz, keep);
            }
          }, [&]() {
            if (i < ti.ndiag && P.diag_mma) {
              // diagonal block: column j is hidden from the tile's position c iff J * 128 + j > pre + r0 / g + c
              const int t0 = sg.pre + sg.r0 / g - J_cur * kBlock;
#pragma unroll 1
              for (int u = 0; u < 4; ++u) {
                const int sh = 32 - 8 * max(0, min(32, lane * 4 + u - t0));   // bits of word 0 that stay clear; of word k 32 k more
                uint32_t w[8];
#pragma unroll
                for (int k = 0; k < 8; ++k) w[k] = __funnelshift_rc(0xfbfbfbfbu, 0u, (uint32_t)max(0, sh + 32 * k));
                bias_row(u, w);
              }
              fence_proxy_async();
              __syncwarp();
            }
          });
          pid_next = fetch_pid(i + 1);   // (it waits for the loads: behind the arrival)
          if constexpr (FP8) {
            if constexpr (WIDEN) {
              if (rc >= 1) live &= mbar_wait(&vraw_empty, (rc - 1) & 1, ctx, 306);
              if (lane == 0 && live) mbar_arrive_expect_tx(&vraw_full, bytes);
              __syncwarp();
              if (pid >= 0 && live) tma_load_3d_hint(sVraw + lane * psz * 128, &map_v, &vraw_full, 0, sg.h, pid * psz, keep);
              ++rc;
            } else {   // the block's F16 copy is one tile
              if (G >= 1) live &= wait_pv(G - 1, 304);  // V stage free
              if (lane == 0 && live) {
                const int row0 = (sg.blk_off + J_cur) * kBlock;
                mbar_arrive_expect_tx(&v_full, kTileBytes);
                tma_load_3d_hint(sV, &map_v, &v_full, 0, sg.h, row0, keep);
                tma_load_3d_hint(sV + 16384, &map_v, &v_full, 64, sg.h, row0, keep);
              }
              __syncwarp();
            }
          } else {
            if (G >= 1) live &= wait_pv(G - 1, 303);  // V stage free
            if (lane == 0 && live) mbar_arrive_expect_tx(&v_full, bytes);
            __syncwarp();
            if (pid >= 0 && live) {
              tma_load_3d_hint(sV + lane * psz * 128, &map_v, &v_full, 0, sg.h, pid * psz, keep);
              tma_load_3d_hint(sV + 16384 + lane * psz * 128, &map_v, &v_full, 64, sg.h, pid * psz, keep);
            }
          }
        } else {
          const int cid = ti.chunk_id[i - T];
          const int row0 = sg.blk_off + cid * 128;
          request_k(kTileBytes, [&]() {
            if (lane == 0 && live) {
              if constexpr (FP8) {   // e4m3 hi | lo, 16 KB each
                tma_load_3d_hint(sK, &map_kbar, &k_full, 0, sg.h, row0, keep);
                tma_load_3d_hint(sK + 16384, &map_kbar_lo, &k_full, 0, sg.h, row0, keep);
              } else {
                tma_load_3d_hint(sK, &map_kbar, &k_full, 0, sg.h, row0, keep);
                tma_load_3d_hint(sK + 16384, &map_kbar, &k_full, 64, sg.h, row0, keep);
              }
            }
          }, [&]() {   // hidden from all positions unless block j is to be corrected
            const uint32_t todo = ti.todo[cid][lane >> 3] >> ((lane * 4) & 31);
#pragma unroll
            for (int u = 0; u < 4; ++u) {
              const uint32_t x = (todo >> u) & 1u ? 0u : 0xfbfbfbfbu;
              bias_row(u, {x, x, x, x, x, x, x, x});
            }
            fence_proxy_async();
            __syncwarp();
          });
          if (G >= 1) live &= wait_pv(G - 1, 305);    // V stage free
          if (lane == 0 && live) {
            if constexpr (WIDEN) mbar_arrive_n(&v_full, 3);
            mbar_arrive_expect_tx(&v_full, kTileBytes);
            tma_load_3d_hint(sV, &map_vbar, &v_full, 0, sg.h, row0, keep);
            tma_load_3d_hint(sV + 16384, &map_vbar, &v_full, 64, sg.h, row0, keep);
          }
          __syncwarp();
        }
      }
      __syncwarp();   // no lane reads the descriptor any more
      if (lane == 0) mbar_arrive(&info_empty[slot]);
    }
  } else if (warp == 5) {
    // =============================== UMMA issuer ===============================
    // The whole warp walks this loop and waits; one elected lane issues.  Outside the elected branches the loop is
    // warp-uniform, which shortens the instruction chain around every MMA: with the loop inside `if (lane == 0)` the
    // issuing thread itself was what the tensor pipe waited for (32768 tokens dense 8429 -> 7993 us, 131072 tokens at 95 %
    // sparsity 11368 -> 10825, FP8 9320 -> 9035, 16 sequences 3702 -> 3556).  The waits' results stay out of it: with a flag per
    // lane that an expired wait clears, `if (leader && live)`, every call was 5 to 10 % slower.
    setmaxnreg_dec<AttnCfg<FP8>::kRegsService>();
    const bool leader = elect_one();
    constexpr int kFmt = FP8 ? 0 : 1;   // kind::f16 operand format of O += P V: 0 = F16, 1 = BF16
    constexpr uint32_t idesc_qk = FP8 ? make_idesc(128, 128, 0, 0, 0, 0)    // kind::f8f6f4, E4M3 x E4M3
                                      : make_idesc(128, 128, 1, 1, 0, 0);
    constexpr uint32_t idesc_pv = make_idesc(128, 128, kFmt, kFmt, 0, 1);
    const uint64_t q_desc = make_smem_desc_sw128(smem_u32(sQ), 16, 1024);
    const uint64_t k_desc = make_smem_desc_sw128(smem_u32(sK), 16, 1024);
    const uint64_t v_desc = make_smem_desc_sw128(smem_u32(sV), 16384, 1024);
    // S = Q K^T of an iteration (chunk: a correction chunk; last: the unit's last one)
    auto issue_qk = [&](bool masked, bool chunk, bool last) {
      if constexpr (FP8) {
        // raw e4m3 operands, 32 elements (= 32 bytes of the swizzled row) per MMA; a correction chunk adds
        // the lo part of the pooled keys on top of the hi part
#pragma unroll
        for (int ks = 0; ks < 4; ++ks) umma_f8_ss(tmem, q_desc + ks * 2, k_desc + ks * 2, idesc_qk, ks > 0);
        if (chunk) {
#pragma unroll
          for (int ks = 0; ks < 4; ++ks) umma_f8_ss(tmem, q_desc + ks * 2, k_desc + (1024 + ks * 2), idesc_qk, 1u);
        }
      } else {
#pragma unroll
        for (int ks = 0; ks < 8; ++ks)   // descriptor addresses count 16 bytes
          umma_f16_ss(tmem, q_desc + ((ks >> 2) * (AttnCfg<FP8>::kQHalf >> 4) + (ks & 3) * 2),
                      k_desc + ((ks >> 2) * 1024 + (ks & 3) * 2), idesc_qk, ks > 0);
      }
      if (masked) {   // the mask as one more k-step (see sBias)
        constexpr uint32_t idesc_bias = make_idesc(128, 128, 1, 1, 0, 0);   // e5m2 x e5m2
        umma_f8_ss(tmem, make_smem_desc_plain(smem_u32(sHot), 128, 256),
                   make_smem_desc_plain(smem_u32(sBias), 128, 256), idesc_bias, 1u);
      }
      umma_commit(&s_done);
      if (last) umma_commit(&q_empty);
    };
    // Look-ahead.  A shared-memory wait that follows a commit in this warp is held until the commit has been taken: from the last
    // slice of O += P V to S = Q K^T (G+1) it took some 500 cycles although K (G+1) had long landed.  So what S = Q K^T (G+1)
    // needs is looked at BEFORE the last slice of P (G) is waited for, across a unit boundary too, and where it is there its
    // MMAs follow those of the last slice without a wait in between.  Without / with it (us): 32768 tokens dense 7760 / 7615,
    // 16384 tokens dense FP8 1503 / 1456, 131072 tokens FP8 7849 / 7715, 8191 tokens FP8 199.3 / 196.2; 131072 and 32768 tokens BF16
    // and 16 sequences within 1 %.  (With P in four slices it gave nothing.)
    uint32_t G = 0;
    bool qk_issued = false;   // S = Q K^T (G) is under way already
    for (int it = 0;; ++it) {
      const int slot = it & 1;
      const TileInfo& ti = info[slot];
      if (!ready_warp(&info_full[slot], (it >> 1) & 1, ctx, 403, &ti.valid)) break;
      const int T = ti.T, ndiag = P.diag_mma ? ti.ndiag : 0;
      const int i0 = ti.it_begin, i1 = ti.it_end;
      if (!qk_issued) mbar_wait(&q_full, it & 1, ctx, 404);
      for (int i = i0; i < i1; ++i, ++G) {
        // S = Q K^T (G).  The S columns are free: O += P V (G-1), which read P out of them, was issued before.
        if (!qk_issued) {
          mbar_wait(&k_full, G & 1, ctx, 405);
          tc_fence_after();
          if (leader) issue_qk(i >= T || i < ndiag, i >= T, i == i1 - 1);
        }
        // O += P V (G)
        mbar_wait(&v_full, G & 1, ctx, 402);
#pragma unroll
        for (int h = 0; h < kPParts - 1; ++h) {   // as each slice of P arrives
          mbar_wait(&p_ready[h], G & 1, ctx, 401);
          tc_fence_after();
          if (leader) {
#pragma unroll
            for (int ks = h ? PSlices<FP8>::end(h - 1) : 0; ks < PSlices<FP8>::end(h); ++ks)
              umma_f16_ts(tmem + 128, tmem + ks * 8, v_desc + ks * 128, idesc_pv, (i > i0) || ks > 0);
          }
        }
        bool masked, chunk, last;
        if (i + 1 < i1) {
          masked = i + 1 >= T || i + 1 < ndiag;
          chunk = i + 1 >= T;
          last = i + 1 == i1 - 1;
          qk_issued = mbar_test(&k_full, (G + 1) & 1);
        } else {
          const TileInfo& tn = info[slot ^ 1];
          qk_issued = mbar_test(&info_full[slot ^ 1], ((it + 1) >> 1) & 1);
          if (qk_issued)
            qk_issued = tn.valid && tn.it_begin < tn.it_end && mbar_test(&q_full, (it + 1) & 1) && mbar_test(&k_full, (G + 1) & 1);
          masked = qk_issued && (tn.it_begin >= tn.T || (P.diag_mma && tn.it_begin < tn.ndiag));
          chunk = qk_issued && tn.it_begin >= tn.T;
          last = qk_issued && tn.it_begin == tn.it_end - 1;
        }
        qk_issued = __all_sync(0xffffffffu, qk_issued);
        mbar_wait(&p_ready[kPParts - 1], G & 1, ctx, 401);
        tc_fence_after();
        if (leader) {
#pragma unroll
          for (int ks = PSlices<FP8>::end(kPParts - 2); ks < 8; ++ks)
            umma_f16_ts(tmem + 128, tmem + ks * 8, v_desc + ks * 128, idesc_pv, 1u);
          umma_commit(&pv_done[G & 1]);
          if (qk_issued) issue_qk(masked, chunk, last);
        }
      }
      __syncwarp();   // no lane reads the descriptor any more
      if (leader) {
        if (i1 == i0) umma_commit(&q_empty);  // nothing to do for this unit: nothing read Q, release it at once
        mbar_arrive(&info_empty[slot]);
      }
    }
  } else {
    // =============================== softmax warpgroup + epilogue ===============================
    setmaxnreg_inc<AttnCfg<FP8>::kRegsSoftmax>();
    const int row = warp * 32 + lane;
    const uint32_t lane_base = tmem + ((uint32_t)(warp * 32) << 16);
    const uint32_t s_addr = lane_base;         // S; P overwrites its first 64 columns
    const uint32_t o_addr = lane_base + 128;
    uint32_t G = 0, rc = 0;   // rc: exact iterations so far (uses of the raw V slot)
    (void)rc;
    const uint64_t stream_pol = l2_policy_evict_first();   // outputs are written once and not read here
#ifdef FP2_PROFILE
    long long pf[16];
    for (int i = 0; i < 16; ++i) pf[i] = 0;
    const long long pf_t0 = clock64();
    long long pf_a, pf_b;
#endif
    for (int it = 0;; ++it) {
      const int slot = it & 1;
      PF_BEGIN();
      const TileInfo& ti = info[slot];
      if (!ready_warp(&info_full[slot], (it >> 1) & 1, ctx, 501, &ti.valid)) break;
      PF_END(0);
      const int T = ti.T;
      const bool dense = ti.dense != 0;
      const int J_hi = ti.sg.J_hi, J_lo = ti.sg.J_lo;
      const int32_t* list = A.blk_idx + ti.sg.off;
      const int r = ti.sg.r0 + row;
      const int pos = ti.sg.pre + r / g;
      // logit multiplier in log2 units.  FP8 (Eq. 15): the MMAs see raw e4m3 values (pooled keys included), so
      // every logit of a row carries q_scale * k_scale; the output carries v_scale.
      float cs_all = P.scale_log2, out_scale = 1.0f;
      if constexpr (FP8) {
        cs_all *= A.q_scale[ti.sg.h * g + r % g] * A.k_scale[ti.sg.h];
        out_scale = A.v_scale[ti.sg.h];
      }
      // The mask bias is -3.3e9 in raw units; with FP8 scales so small that this is no longer far below every
      // visible logit of the row, the warp masks in TMEM as well.
      bool weak_bias = false;
      if constexpr (FP8) weak_bias = __any_sync(0xffffffffu, !(cs_all * 3.0e9f > 256.f));
      const bool row_ok = row < ti.sg.nrows;   // else padding: whatever queries follow, those of other sequences among them
      float m = -INFINITY, l = 0.f;
      // block id of the next exact iteration, fetched one iteration ahead
      const int i0 = ti.it_begin, i1 = ti.it_end;
      int J_next = (!dense && i0 < T) ? list[T - 1 - i0] : 0;
      for (int i = i0; i < i1; ++i, ++G) {
        // iteration kind and masks
        bool need_mask = false;
        int tok_lim = 1 << 30;     // exact block: columns j with j <= tok_lim are visible
        uint32_t cm0 = 0xffffffffu, cm1 = 0xffffffffu, cm2 = 0xffffffffu, cm3 = 0xffffffffu;
        float shift = 0.f;
        if (i < T) {
          int J = dense ? J_hi - i : J_next;
          if (!dense && i + 1 < T) J_next = list[T - 2 - i];
          J = max(0, min(J, J_hi));
          need_mask = J >= J_lo && (!P.diag_mma || weak_bias);   // else the causal mask is in the logits already
          tok_lim = pos - J * kBlock;
        } else {
          shift = 7.0f;  // log2(128): one pooled row stands for a full block (Eq. 6); the todo mask is in the logits already
          if (weak_bias) {
            const int c = ti.chunk_id[i - T];
            cm0 = ti.todo[c][0];
            cm1 = ti.todo[c][1];
            cm2 = ti.todo[c][2];
            cm3 = ti.todo[c][3];
            need_mask = true;
          }
        }
        if constexpr (WIDEN) {
          // Exact iteration: widen this iteration's raw e4m3 V tile (exactly) into the F16 V stage before looking
          // at the logits.  128 threads take ~900 cycles (the copy is bound by shared-memory bandwidth next to the
          // other CTA's MMAs); one or two dedicated warps were slower than the time they have, between
          // O += P V (G-1) freeing the stage and the first slice of P (G) needing it.
          if (i < T) {
            mbar_wait(&vraw_full, rc & 1, ctx, 603);
            if (G >= 1) wait_pv(G - 1, 602);
            widen_tile_f16(sVraw, sV, tid, 128);
            fence_proxy_async();
            __syncwarp();
            if (lane == 0) {   // (no barrier between the warps: after an abort one of them may have left)
              mbar_arrive(&vraw_empty);
              mbar_arrive(&v_full);
            }
            ++rc;
          }
        }
        PF_BEGIN();
        mbar_wait(&s_done, G & 1, ctx, 502);
        PF_END(i == i0 ? 1 : (i < T ? 2 : 3));
#ifdef FP2_PROFILE
        pf[i == i0 ? 8 : (i < T ? 9 : 10)] += 1;
#endif
        tc_fence_after();
        if (need_mask) mask_row(s_addr, tok_lim, cm0, cm1, cm2, cm3);
        PF_END(4);
        uint32_t x[128];
        const float mx = fmaf(row_load_max(s_addr, x), cs_all, shift);  // cs > 0: scaling commutes with the maximum
        const float m_new = fmaxf(m, mx);
        // lazy rescale: only when some row of the warp moved its maximum by more than 2^8.  O is at rest: the
        // MMAs complete in issue order, so S (G) in TMEM means O += P V (G-1) has been added.  Padding rows have no say (their
        // probabilities may overflow, which stays in their own rows): when a row is rescaled decides how its probabilities round,
        // and that must not hang on what the batch holds beside its sequence.
        if (__any_sync(0xffffffffu, row_ok && m_new > m + 8.0f)) {
          const float f = (m == -INFINITY) ? 0.f : ex2(m - m_new);
          if (i > i0) {
#pragma unroll 1
            for (int k = 0; k < 4; ++k) {
              uint32_t rr[32];
              tmem_ld32(o_addr + k * 32, rr);
              tmem_wait_ld();
#pragma unroll
              for (int j = 0; j < 32; ++j) rr[j] = __float_as_uint(__uint_as_float(rr[j]) * f);
              tmem_st32(o_addr + k * 32, rr);
            }
          }
          l *= f;
          m = m_new;
        }
        // a row with nothing visible so far has m = -inf and only -inf logits: exponent against 0 -> zeros
        const float neg_m = (m == -INFINITY) ? shift : shift - m;
        l += row_exp<FP8>(x, s_addr, cs_all, neg_m, &p_ready[0]);
        tmem_wait_st();
        tc_fence_before();
        mbar_arrive(&p_ready[kPParts - 1]);
        PF_END(5);
      }
      // ------------------------------ epilogue ------------------------------
      PF_BEGIN();
      const SegInfo& sg = ti.sg;
      const float inv = l > 0.f ? out_scale / l : 0.f;
      const bool have_o = i1 > i0;
      const size_t tok = (size_t)sg.q_tok0 + r / g;
      const int head = sg.h * g + r % g;
      __nv_bfloat16* orow = A.out + (tok * P.num_q_heads + head) * kHeadDim;
      if (have_o) {
        wait_pv(G - 1, 503);   // O += P V of the unit's last iteration
        tc_fence_after();
      }
      PF_END(6);
      if (ti.parts > 1) {
        // one part of a split segment (Eq. 18): leave (O, m, l) unnormalised for the merge kernel
        float* prow = A.part_o + ((size_t)ti.slot * 128 + row) * 128;
        if (have_o) {
#pragma unroll 1
          for (int k = 0; k < 4; ++k) {
            uint32_t a0[32];
            tmem_ld32(o_addr + k * 32, a0);
            tmem_wait_ld();
#pragma unroll
            for (int j = 0; j < 4; ++j) st_global_v8(prow + k * 32 + j * 8, &a0[j * 8], stream_pol);
          }
        }
        A.part_ml[(size_t)ti.slot * 128 + row] = make_float2(have_o ? m : -INFINITY, have_o ? l : 0.f);
        tc_fence_before();
        mbar_arrive(&info_empty[slot]);
        continue;
      }
#pragma unroll 1
      for (int k = 0; k < 4; ++k) {
        uint32_t a0[32];
        if (have_o) {
          tmem_ld32(o_addr + k * 32, a0);
          tmem_wait_ld();
        }
        uint32_t o[16];
#pragma unroll
        for (int j = 0; j < 16; ++j) {
          const float v0 = have_o ? __uint_as_float(a0[2 * j]) * inv : 0.f;
          const float v1 = have_o ? __uint_as_float(a0[2 * j + 1]) * inv : 0.f;
          o[j] = pack_bf16x2(v0, v1);
        }
        if (row_ok) {   // 32-byte stores: every instruction writes whole sectors
          st_global_v8(orow + k * 32, &o[0], stream_pol);
          st_global_v8(orow + k * 32 + 16, &o[8], stream_pol);
        }
      }
      if (row_ok && A.lse != nullptr)
        A.lse[(size_t)head * P.total_q + tok] = (m + log2f(l)) * 0.6931471805599453f;
      tc_fence_before();
      mbar_arrive(&info_empty[slot]);
      PF_END(7);
    }
#ifdef FP2_PROFILE
    pf[15] = clock64() - pf_t0;
    if (tid == 0 && A.prof)
      for (int i = 0; i < 16; ++i) A.prof[(size_t)blockIdx.x * 16 + i] = pf[i];
#endif
  }
  leave_cta(ctx, &drain_bar, warp == 5);
  if (warp == 5) tmem_dealloc(tmem, 256);
}

}  // namespace fp2
