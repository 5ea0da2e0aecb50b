// Shared device-side definitions: segment table entries, kernel parameter block, compile-time shape.
#pragma once
#include <stdint.h>

namespace fp2 {

constexpr int kHeadDim = 128;     // d
constexpr int kBlock = 128;       // B: KV tokens per selection block (Sec. 4.1)
constexpr int kTileRows = 128;    // packed query rows per tile (kBlockM, Sec. 4.1)
constexpr int kMaxBlocks = 4096;  // KV blocks per sequence the kernels are compiled for (512K tokens)
constexpr int kMaxChunks = kMaxBlocks / 128;
// Query tiles by TMA.  Under PackGQA (Eq. 13) the packed rows of a tile are consecutive (token, head) pairs of one KV head's
// group, so the box [128 bytes, g heads, tokens] that starts at the tile's first token holds them all, in packed order, the
// first one r0 % g rows into it.  Where g does not divide 128 the box lands that many rows in front of the tile's place in
// shared memory (the 128-byte swizzle goes by the address, so the tile itself sits as the MMA reads it) and its overhang on
// padding: at most kQLeadRows rows in front and kQTailRows behind.
constexpr int kQLeadRows = 8;
constexpr int kQTailRows = 16;
constexpr int kCountBuckets = 128;   // work-order classes per KV head (selected-block count, see order_bucket)

// One (sequence, KV head, tile) segment; built on the host by the planner.
struct SegInfo {
  int32_t b, h, t;
  int32_t nrows;    // real packed rows in the tile (<= 128)
  int32_t q_tok0;   // cu_seqlens_q[b]
  int32_t r0;       // first packed row of the tile
  int32_t pre;      // cached prefix length Lk - Lq
  int32_t Lk;
  int32_t J_lo;     // block of the first row's absolute position
  int32_t J_hi;     // block of the last row's absolute position (candidates are 0..J_hi)
  int32_t blk_off;  // first row of this sequence in the pooled-mean arrays
  int32_t seg;      // index of this segment in segment order
  int64_t off;      // seg_offset: start of this segment's list in blk_idx
  __host__ __device__ int h_seg() const { return seg; }
};
static_assert(sizeof(SegInfo) == 56, "SegInfo layout");

struct DevParams {
  int32_t num_q_heads, num_kv_heads, group;
  int32_t page_size, pages_per_block, max_pages_per_seq, num_pages;
  int32_t sink_blocks, window_blocks, use_correction;
  int32_t num_seqs, nseg, nblk_tot, total_q;
  int32_t fp8;
  int32_t q_box;     // 1: the boxes around one packed tile (q_box_tok tokens) and around two adjacent ones (q_box2_tok) fit the
                     //    padding: attention kernel and paired scorer (both dtypes) fetch query tiles by TMA.  Not so for
                     //    group sizes such as 11, 12 or 48, whose boxes reach further in front of a tile or behind it
  int32_t q_box_tok, q_box2_tok;   // 128 / g tokens where g divides 128, else floor((g - 1 + 127) / g) + 1; 256 rows likewise
  int32_t q_raw_tma; // 1: FP8 plans whose box fits the scorer's raw staging slot: the scorer fetches query tiles by TMA
  int32_t diag_mma;  // 1: a tile spans at most 32 positions (g >= 4), so the causal mask of a diagonal block can ride
                     //    on a K = 32 one-hot MMA step in the attention kernel
  float alpha;
  float scale_log2;  // softmax scale * log2(e)
};

}  // namespace fp2
