// Block-mean pooling (Eq. 5; Algorithm 1 line 2): kbar_J, vbar_J = mean over the real tokens of KV block J,
// read through the page table (Eq. 22).  HBM-bound: K and V are read exactly once with 16-byte loads,
// 256-byte (BF16) or 128-byte (FP8) contiguous per token row, fp32 accumulation.
//
// Outputs, all BF16 [nblk_tot, Hkv, 128]:
//   kbar_hi = bf16(mean k), kbar_lo = bf16(mean k - kbar_hi)   (hi + lo carries ~16 mantissa bits for the scorer)
//   vbar    = bf16(mean v)
// kbar_hi and vbar double as the operands of the correction chunks in the attention kernel.
// FP8 inputs: the three arrays hold F16 instead of BF16: kbar_hi / kbar_lo = F16 pair of the de-scaled mean (mean
// of raw values x k_scale) for the scorer, vbar = f16(mean of RAW v) -- v_scale is applied to the attention
// output.  Two more arrays, e4m3 [nblk_tot, Hkv, 128] each, hold the mean of the RAW keys as a hi + lo pair
// (hi = e4m3(mean), lo = e4m3(mean - hi): ~8 mantissa bits together) for the correction chunks of the attention
// kernel, whose S = Q K^T runs on raw e4m3 operands.
#pragma once
#include <cuda_bf16.h>
#include <cuda_fp16.h>
#include <cuda_fp8.h>
#include "common.cuh"
#include "ptx.cuh"
#include "split_kv.cuh"   // pack_split

namespace fp2 {

template <bool FP8>
__device__ __forceinline__ void accum16(const uint4& v, float* acc) {
  if constexpr (!FP8) {
    const __nv_bfloat162* p = reinterpret_cast<const __nv_bfloat162*>(&v);
#pragma unroll
    for (int i = 0; i < 4; ++i) {
      float2 f = __bfloat1622float2(p[i]);
      acc[2 * i] += f.x;
      acc[2 * i + 1] += f.y;
    }
  } else {
    const __nv_fp8x2_storage_t* p = reinterpret_cast<const __nv_fp8x2_storage_t*>(&v);
#pragma unroll
    for (int i = 0; i < 8; ++i) {
      __half2_raw h = __nv_cvt_fp8x2_to_halfraw2(p[i], __NV_E4M3);
      float2 f = __half22float2(*reinterpret_cast<__half2*>(&h));
      acc[2 * i] += f.x;
      acc[2 * i + 1] += f.y;
    }
  }
}

// One pooled mean -> the operand formats the scorer and the correction chunks read (see the head of the file).
template <bool FP8>
__device__ __forceinline__ void write_pooled(int which, float mean, size_t o, int h, const float* k_scale,
                                             __nv_bfloat16* __restrict__ kbar_hi, __nv_bfloat16* __restrict__ kbar_lo,
                                             __nv_bfloat16* __restrict__ vbar, uint8_t* __restrict__ kbar8_hi,
                                             uint8_t* __restrict__ kbar8_lo) {
  if constexpr (FP8) {
    if (which == 0) {
      // the attention kernel multiplies raw e4m3 queries with this pair in one FP8 MMA group each
      const __nv_fp8_storage_t hi8 = __nv_cvt_float_to_fp8(mean, __NV_SATFINITE, __NV_E4M3);
      const float hi8f = __half2float(__half(__nv_cvt_fp8_to_halfraw(hi8, __NV_E4M3)));
      kbar8_hi[o] = hi8;
      kbar8_lo[o] = __nv_cvt_float_to_fp8(mean - hi8f, __NV_SATFINITE, __NV_E4M3);
      mean *= k_scale[h];
    }
    const __half hi16 = __float2half_rn(mean);
    if (which == 0) {
      reinterpret_cast<__half*>(kbar_hi)[o] = hi16;
      reinterpret_cast<__half*>(kbar_lo)[o] = __float2half_rn(mean - __half2float(hi16));
    } else {
      reinterpret_cast<__half*>(vbar)[o] = hi16;
    }
  } else {
    const __nv_bfloat16 hi16 = __float2bfloat16_rn(mean);
    if (which == 0) {
      kbar_hi[o] = hi16;
      kbar_lo[o] = __float2bfloat16_rn(mean - __bfloat162float(hi16));
    } else {
      vbar[o] = hi16;
    }
  }
}

// 1-D grid of nblk_tot * Hkv * 2 CTAs: (K or V) fastest, then the KV head, then the block, so CTAs that run
// together read neighbouring pieces of the same token rows.  One CTA pools one operand of one (block, head):
// 128 token rows of 256 B (BF16) / 128 B (FP8).  256 threads, every load of a thread issued before the first
// use; small enough in registers for four CTAs per SM, which is what hides the page-table -> data dependency.
template <bool FP8>
__global__ void __launch_bounds__(256, 4) pool_kv_kernel(const uint8_t* k_cache,
                                                         const uint8_t* v_cache,
                                                         const int32_t* page_table,
                                                         const int32_t* __restrict__ plan_lk,  // [ns], the plan's copy
                                                         const int32_t* __restrict__ blk_off,  // [ns+1]
                                                         const float* k_scale,
                                                         const float* v_scale, DevParams P,
                                                         __nv_bfloat16* __restrict__ kbar_hi,
                                                         __nv_bfloat16* __restrict__ kbar_lo,
                                                         __nv_bfloat16* __restrict__ vbar,
                                                         uint8_t* __restrict__ kbar8_hi,
                                                         uint8_t* __restrict__ kbar8_lo,
                                                         const int32_t* carry,
                                                         int* __restrict__ status) {
  constexpr int ROW_BYTES = FP8 ? 128 : 256;
  constexpr int CHUNKS = ROW_BYTES / 16;       // 16-byte chunks per token row
  constexpr int EPC = FP8 ? 16 : 8;            // elements per chunk
  constexpr int ROWS_PER_PASS = 256 / CHUNKS;  // 16 (bf16) or 32 (fp8)
  constexpr int PASSES = kBlock / ROWS_PER_PASS;

  __shared__ float red[ROWS_PER_PASS][kHeadDim + 4];
  pdl_trigger();
  pdl_wait();

  const int which = blockIdx.x & 1;            // 0: K, 1: V
  const int bh = blockIdx.x >> 1;
  const int gblk = bh / P.num_kv_heads, h = bh % P.num_kv_heads;
  // sequence of this pooled block: binary search in blk_off
  int lo = 0, hi = P.num_seqs;
  while (hi - lo > 1) {
    int mid = (lo + hi) >> 1;
    if (blk_off[mid] <= gblk) lo = mid; else hi = mid;
  }
  const int b = lo, J = gblk - blk_off[b];
  // chunked prefill: the means of the first carry[3 b + 2] blocks of this sequence were carried over from the
  // previous chunk's workspace (pool_carry_kernel) and are not computed again
  if (carry != nullptr && J < carry[3 * b + 2]) return;
  // The length comes from the plan's table (validated on the host when the plan was made), like every other piece
  // of geometry: a block of the pooled arrays always has between 1 and 128 real tokens.
  const int Lk = plan_lk[b];
  const int ntok = min(kBlock, Lk - J * kBlock);
  const int chunk = threadIdx.x % CHUNKS, rg = threadIdx.x / CHUNKS;
  const int32_t* pt = page_table + (size_t)b * P.max_pages_per_seq;
  const size_t row_stride = (size_t)P.num_kv_heads * ROW_BYTES;
  const uint8_t* cache = which ? v_cache : k_cache;

  uint4 dv[PASSES];
#pragma unroll
  for (int ps = 0; ps < PASSES; ++ps) {
    const int tl = ps * ROWS_PER_PASS + rg;
    dv[ps] = make_uint4(0, 0, 0, 0);   // zero bit patterns add 0 in both encodings
    if (tl < ntok) {
      const int j = J * kBlock + tl;
      const int pid = pt[j / P.page_size];
      if (pid < 0 || pid >= P.num_pages) {
        // a page id outside the pool: nothing is read for this token (it counts as zeros) and the call is flagged
        atomicOr(status + ST_BAD_LIST, 2);
      } else {
        const size_t slot = (size_t)pid * P.page_size + (j % P.page_size);
        dv[ps] = __ldg(reinterpret_cast<const uint4*>(cache + slot * row_stride + (size_t)h * ROW_BYTES + chunk * 16));
      }
    }
  }
  float acc[EPC];
#pragma unroll
  for (int i = 0; i < EPC; ++i) acc[i] = 0.f;
#pragma unroll
  for (int ps = 0; ps < PASSES; ++ps) accum16<FP8>(dv[ps], acc);
#pragma unroll
  for (int i = 0; i < EPC; ++i) red[rg][chunk * EPC + i] = acc[i];
  __syncthreads();
  if (threadIdx.x < kHeadDim) {
    const int c = threadIdx.x;
    float s = 0.f;
#pragma unroll
    for (int r = 0; r < ROWS_PER_PASS; ++r) s += red[r][c];
    const size_t o = ((size_t)gblk * P.num_kv_heads + h) * kHeadDim + c;
    write_pooled<FP8>(which, s / (float)ntok, o, h, k_scale, kbar_hi, kbar_lo, vbar, kbar8_hi, kbar8_lo);
  }
}

// The same pooling with one CTA per (block, K or V) over ALL KV heads: a token's row of the cache is
// Hkv x 128 elements contiguous, so the CTA streams 128 whole rows (256 KB for 8 BF16 heads) behind ONE look-up of
// the block's page ids instead of one dependent look-up per 32 KB.  Used when the row's 16-byte chunks divide 256
// (Hkv a power of two, at most 16 BF16 / 32 FP8 heads).  Thread t owns chunk t mod C of the row and the tokens
// t / C, t / C + G, ... (G = 256 / C token groups): four 16-byte loads in flight per thread and batch, four CTAs per
// SM, fp32 accumulation, one shared-memory reduction over the G groups.  Page sizes are powers of two, so the slot
// of a token takes a shift and a mask (a division per load made the kernel ALU-bound: 143 -> 110 us at 128K).
// Measured at 131072 tokens, 8 BF16 heads: 93 us for 537 MB = 5.8 TB/s; a bare streaming read reaches 6.8 TB/s.
template <bool FP8>
__global__ void __launch_bounds__(256, 4) pool_rows_kernel(const uint8_t* k_cache,
                                                           const uint8_t* v_cache,
                                                           const int32_t* page_table,
                                                           const int32_t* __restrict__ plan_lk,
                                                           const int32_t* __restrict__ blk_off,
                                                           const float* k_scale,
                                                           const float* v_scale, DevParams P,
                                                           __nv_bfloat16* __restrict__ kbar_hi,
                                                           __nv_bfloat16* __restrict__ kbar_lo,
                                                           __nv_bfloat16* __restrict__ vbar,
                                                           uint8_t* __restrict__ kbar8_hi,
                                                           uint8_t* __restrict__ kbar8_lo,
                                                           const int32_t* carry,
                                                           int* __restrict__ status) {
  constexpr int CH = FP8 ? 8 : 16;             // 16-byte chunks per head row
  constexpr int EPC = FP8 ? 16 : 8;            // elements per chunk
  constexpr int BATCH = 4;                     // loads in flight per thread; four CTAs per SM overlap each other's set-up and reduction
  __shared__ float red[256 * EPC];             // [token group][chunk][element]
  __shared__ int32_t pids[kBlock / 8];         // page ids of the block (page size >= 8)

  pdl_trigger();
  const int which = blockIdx.x & 1;            // 0: K, 1: V
  const int gblk = blockIdx.x >> 1;
  int lo = 0, hi = P.num_seqs;
  while (hi - lo > 1) {
    int mid = (lo + hi) >> 1;
    if (blk_off[mid] <= gblk) lo = mid; else hi = mid;
  }
  const int b = lo, J = gblk - blk_off[b];   // (the plan's table so far: not written by any kernel)
  pdl_wait();
  if (carry != nullptr && J < carry[3 * b + 2]) return;   // carried over from the previous chunk (pool_carry_kernel)
  const int Lk = plan_lk[b];
  const int ntok = min(kBlock, Lk - J * kBlock);
  const int psz = P.page_size, ppb = P.pages_per_block;
  const int psz_log2 = 31 - __clz(psz);        // page sizes are powers of two: shifts and masks, no divisions per load
  if ((int)threadIdx.x < ppb) {
    int pid = -1;
    if ((int)threadIdx.x * psz < ntok) {
      pid = page_table[(size_t)b * P.max_pages_per_seq + J * ppb + threadIdx.x];
      if (pid < 0 || pid >= P.num_pages) {   // outside the pool: its tokens count as zeros, the call is flagged
        atomicOr(status + ST_BAD_LIST, 2);
        pid = -1;
      }
    }
    pids[threadIdx.x] = pid;
  }
  __syncthreads();

  const int C = P.num_kv_heads * CH;           // chunks per token row; divides 256
  const int G = 256 / C;
  const int chunk = threadIdx.x % C, tg = threadIdx.x / C;
  const int per = kBlock / G;                  // tokens of this thread
  const size_t row_bytes = (size_t)C * 16;
  const uint8_t* cache = which ? v_cache : k_cache;
  float acc[EPC];
#pragma unroll
  for (int i = 0; i < EPC; ++i) acc[i] = 0.f;
  for (int i0 = 0; i0 < per; i0 += BATCH) {
    // every load of the batch is issued unconditionally (a token that is not there reads the start of the cache
    // instead and is replaced by zeros afterwards), so that all of them are in flight before the first use
    uint4 dv[BATCH];
    bool ok[BATCH];
#pragma unroll
    for (int u = 0; u < BATCH; ++u) {
      const int tl = tg + (i0 + u) * G;        // consecutive token groups interleave: the CTA reads G rows at a time
      const int pid = pids[min(tl, kBlock - 1) >> psz_log2];
      ok[u] = i0 + u < per && tl < ntok && pid >= 0;
      const size_t off = ok[u] ? (((size_t)pid << psz_log2) + (size_t)(tl & (psz - 1))) * row_bytes + chunk * 16 : 0;
      dv[u] = __ldg(reinterpret_cast<const uint4*>(cache + off));
    }
#pragma unroll
    for (int u = 0; u < BATCH; ++u) {
      if (!ok[u]) dv[u] = make_uint4(0, 0, 0, 0);   // zero bit patterns add 0 in both encodings
      accum16<FP8>(dv[u], acc);
    }
  }
#pragma unroll
  for (int i = 0; i < EPC; ++i) red[(tg * C + chunk) * EPC + i] = acc[i];
  __syncthreads();
  const int nout = C * EPC;                    // Hkv x 128 means
  for (int o = threadIdx.x; o < nout; o += 256) {
    float sum = 0.f;
    for (int r = 0; r < G; ++r) sum += red[r * nout + o];
    const int h = o / kHeadDim;
    write_pooled<FP8>(which, sum / (float)ntok, (size_t)gblk * nout + o, h, k_scale, kbar_hi, kbar_lo, vbar, kbar8_hi,
                      kbar8_lo);
  }
}

// ----------------------------------------------------------------------------------------
// Work ordering (Sec. 3.3 "Sparsity-Aware Load Balancing", Eq. 21): segments sorted KV-head-major, then by
// descending block count, by a counting sort on the device.  Counts below 64 are classes of their own, larger ones fall
// into eight classes per power of two: heaviest-first needs no finer order, and with 128 classes per head (1024 before)
// the last kernel finds its own offsets instead of waiting for a kernel that scans the histogram (3 us at 64 segments,
// 9 us at 44000).  Order inside a class is arbitrary; it only changes which CTA runs a segment,
// never a result.
// ----------------------------------------------------------------------------------------
__device__ __forceinline__ int order_bucket(int h, int count) {
  int c = max(count, 0);
  if (c >= 64) {
    const int e = 31 - __clz(c);                                    // 6 .. : c in [2^e, 2^(e+1))
    c = min(64 + (e - 6) * 8 + ((c >> (e - 3)) & 7), kCountBuckets - 1);
  }
  return h * kCountBuckets + (kCountBuckets - 1 - c);
}

// V of FP8 plans as F16 (exact), [nblk_tot * 128, Hkv, 128]: the attention kernel multiplies 16-bit probabilities with it and
// reads every V tile many times; widened in the kernel, every time, it took the softmax warpgroup ~900 cycles per block.
// One CTA per 32 tokens of a block, all KV heads (a quarter block: short prompts have few blocks); rows past the end of the
// sequence are zeros.  Bandwidth-bound: 1 byte read, 2 written per element.  The loads of a batch are unconditional, as in
// pool_rows_kernel: behind a branch each they went out one at a time (8192 tokens, 4 heads: 27 us, now 8; 245000 tokens, 8 heads: 145 us = 5.2 TB/s).
constexpr int kWidenTokens = 32;
__device__ __forceinline__ void widen_v_part(const uint8_t* v_cache, const int32_t* page_table, const int32_t* plan_lk,
                                             const int32_t* blk_off, const DevParams& P, int part, __half* v16, int* status) {
  __shared__ int32_t pids[kWidenTokens / 8];   // page ids of the tokens (page size >= 8), -1: nothing to read
  const int gblk = part / (kBlock / kWidenTokens), tok0 = part % (kBlock / kWidenTokens) * kWidenTokens;
  int lo = 0, hi = P.num_seqs;
  while (hi - lo > 1) {
    const int mid = (lo + hi) >> 1;
    if (blk_off[mid] <= gblk) lo = mid; else hi = mid;
  }
  const int b = lo, j0 = (gblk - blk_off[b]) * kBlock + tok0;   // first token of the part
  const int ntok = min(kWidenTokens, plan_lk[b] - j0);
  const int psz = P.page_size, psz_log2 = 31 - __clz(psz);
  const int first_page = j0 >> psz_log2;
  if ((int)threadIdx.x < kWidenTokens / 8) {
    int pid = -1;
    const int page = first_page + (int)threadIdx.x;
    if ((page << psz_log2) < j0 + ntok) {
      pid = page_table[(size_t)b * P.max_pages_per_seq + page];
      if (pid < 0 || pid >= P.num_pages) {   // outside the pool: its tokens count as zeros, the call is flagged
        atomicOr(status + ST_BAD_LIST, 2);
        pid = -1;
      }
    }
    pids[threadIdx.x] = pid;
  }
  __syncthreads();
  const int C = P.num_kv_heads * 8;            // 16-byte chunks per token row
  const uint4* src = reinterpret_cast<const uint4*>(v_cache);
  uint4* dst = reinterpret_cast<uint4*>(v16) + ((size_t)gblk * kBlock + tok0) * C * 2;
  constexpr int BATCH = 4;
  const int n = kWidenTokens * C;              // a multiple of 256
  for (int i0 = threadIdx.x; i0 < n; i0 += BATCH * 256) {
    uint4 v[BATCH];
    bool ok[BATCH];
#pragma unroll
    for (int u = 0; u < BATCH; ++u) {
      const int i = min(i0 + u * 256, n - 1), tl = i / C, j = j0 + tl;
      const int pid = pids[(j >> psz_log2) - first_page];
      ok[u] = tl < ntok && pid >= 0;
      const size_t off = ok[u] ? (((size_t)pid << psz_log2) + (j & (psz - 1))) * C + (i - tl * C) : 0;
      v[u] = __ldg(src + off);
    }
#pragma unroll
    for (int u = 0; u < BATCH; ++u) {
      const int i = i0 + u * 256;
      if (i >= n) break;
      if (!ok[u]) v[u] = make_uint4(0, 0, 0, 0);
      dst[2 * (size_t)i] = make_uint4(e4m3x2_to_f16x2(v[u].x), e4m3x2_to_f16x2(v[u].x >> 16), e4m3x2_to_f16x2(v[u].y),
                                      e4m3x2_to_f16x2(v[u].y >> 16));
      dst[2 * (size_t)i + 1] = make_uint4(e4m3x2_to_f16x2(v[u].z), e4m3x2_to_f16x2(v[u].z >> 16), e4m3x2_to_f16x2(v[u].w),
                                          e4m3x2_to_f16x2(v[u].w >> 16));
    }
  }
}

// First kernel of an attention call.  The first n_clear CTAs (256 threads) clear histogram and cursors (nb2 words) and the
// work counter block (16 words); the others, of FP8 plans, widen 32 tokens of V each.
__global__ void __launch_bounds__(256) attn_prepare_kernel(int32_t* __restrict__ hist, int nb2, int32_t* __restrict__ counter,
                                                           int n_clear, const uint8_t* v_cache, const int32_t* page_table,
                                                           const int32_t* __restrict__ plan_lk,
                                                           const int32_t* __restrict__ blk_off, DevParams P, __half* v16,
                                                           int* status) {
  pdl_trigger();
  pdl_wait();
  if ((int)blockIdx.x >= n_clear) {
    widen_v_part(v_cache, page_table, plan_lk, blk_off, P, (int)blockIdx.x - n_clear, v16, status);
    return;
  }
  const int i = blockIdx.x * blockDim.x + threadIdx.x;
  if (i < nb2) hist[i] = 0;
  if (i < 16) counter[i] = 0;
}

// Where every segment has a worker of its own (nseg <= workers) all of them start at once: there is nothing to sort, the order
// is the segments' own.  Sorted / so: select + sparse, 768 tokens FP8 35.5 / 33.3 us, 2370 tokens 41.5 / 40.3, 2048 tokens 34.4 /
// 32.9; dense, 839 tokens 22.9 / 22.1.
__global__ void order_hist_kernel(const SegInfo* __restrict__ segs, const int32_t* count, int nseg, int workers,
                                  int32_t* __restrict__ hist) {
  pdl_trigger();
  const int s = blockIdx.x * blockDim.x + threadIdx.x;
  const int h = s < nseg ? segs[s].h : 0, J = s < nseg ? segs[s].J_hi : 0;   // the plan's table: not written by any kernel
  pdl_wait();
  if (s >= nseg || nseg <= workers) return;
  atomicAdd(&hist[order_bucket(h, count ? count[s] : J + 1)], 1);
}

// Places.  A long segment that starts late is what everybody waits for at the end, and KV-head-major order starts the last
// head's long ones late.  So segments longer than 1 / kLongShare of a worker's share of all listed blocks come first, heads
// mixed, longest first; the others follow KV-head-major (the K / V of one head stay in L2), in descending order too.  With
// many segments per worker hardly any is that long and the order is KV-head-major; with few the heads run side by side
// whatever the order is.  Whole calls, KV-head-major throughout / shares of 1/4 / 1/8 / 1/16, in turn: the last 8192 of 131072
// tokens 1514 / 1347 / 1375 / 1408 us, FP8 1204 / 1075 / 1084 / 1088, 32768 tokens 1778 / 1780 / 1731 / 1759, 8191 tokens FP8
// 206.5 / 201.7 / 196.4 / 196.2; 131072 tokens, and 15616 tokens with 32 heads on 4, the same.
// Every CTA of 256 threads adds the histogram up for itself (Hkv x 128 counts, in L2): column sums and their prefix give the
// long segments' places, and the number of long segments per head (head_long, Hkv words of shared memory) the start of each
// head.  Above kMaxLongHeads heads (32 KB; the launch's limit with the static arrays is 48) the order is KV-head-major
// throughout: with 28 segments per worker and more the end of the call is a small part of it.
constexpr int kLongShare = 8;
constexpr int kMaxLongHeads = 8192;
__device__ __forceinline__ int class_min_count(int c) {   // smallest block count of class c (0 .. kCountBuckets - 1)
  const int v = kCountBuckets - 1 - c;
  return v < 64 ? v : (8 + (v & 7)) << ((v - 64) / 8 + 3);
}
// Cutting (Eq. 18).  A segment longer than a worker's share outlasts the rest even when it starts first (the last 8192 of
// 131072 tokens: one list of 408 blocks against a share of 287).  Calls that can have such segments (template parameter CUT, see
// fp2_plan_create) ask for units instead of segments: if the longest class exceeds kCutFrom shares, segments longer than half a
// share become parts of about that length, longest classes first while their partial results fit into max_slots, and the
// merge kernel of the split path puts them together.  That call 1133 -> 1049 us, with a list of 466 blocks against a share of 382
// 1380 -> 1328; where the longest list is below a share nothing is cut.  Against attention in 64 bits the parts' result is as
// far off as the uncut one (rel 1.8059e-3 / 1.8066e-3, 100001 tokens 1.7861e-3 / 1.8029e-3, FP8 1.66254e-3 / 1.66258e-3).
// unit_split[w]: see pack_split; *n_units: units; seg_split, split_list, *n_split: what the merge kernel reads.
struct ClassScan {   // exclusive prefix over the classes, four per lane of a warp
  int before[4], total;
  __device__ __forceinline__ ClassScan(const int (&c)[4], int lane) {
    const int mine = c[0] + c[1] + c[2] + c[3];
    int incl = mine;
#pragma unroll
    for (int o = 1; o < 32; o <<= 1) {
      const int y = __shfl_up_sync(0xffffffffu, incl, o);
      if (lane >= o) incl += y;
    }
    int run = incl - mine;
#pragma unroll
    for (int i = 0; i < 4; ++i) {
      before[i] = run;
      run += c[i];
    }
    total = __shfl_sync(0xffffffffu, incl, 31);
  }
};
constexpr float kCutFrom = 1.0f;
constexpr int kCutMin = 64;           // blocks of a segment below which cutting costs more (Q tile, partial result, merge) than it gives
constexpr int kMaxCuts = 8;           // parts of a segment
struct CutLists {
  int32_t* unit_split;
  int32_t* seg_split;
  int32_t* split_list;
  int32_t* n_units;
  int32_t* n_split;
  int32_t max_slots;
};
template <bool CUT>
__global__ void __launch_bounds__(256) order_scatter_kernel(const SegInfo* __restrict__ segs, const int32_t* count, int nseg,
                                                            int per_head, int num_heads, int workers, const int32_t* hist,
                                                            int32_t* __restrict__ cursor, int32_t* __restrict__ order,
                                                            CutLists cut) {
  static_assert(kCountBuckets == 128, "thread t adds up class t mod 128; a lane of the scan takes four classes");
  extern __shared__ int32_t head_long[];       // [num_heads] long segments per head (up to kMaxLongHeads heads, else unused)
  __shared__ int32_t col[2][kCountBuckets];    // segments per class over all heads (two halves of the heads)
  __shared__ int32_t before[kCountBuckets];    // units of the long segments of the classes in front of this one
  __shared__ int32_t parts[kCountBuckets];      // parts per segment of the class
  __shared__ int32_t slots_before[kCountBuckets], cuts_before[kCountBuckets];   // partial-result slots, cut segments likewise
  __shared__ int s_first_short, s_num_long;    // first class that is not long; units of the long segments
  pdl_trigger();
  const int t = threadIdx.x, lane = t & 31, warp = t >> 5;
  const int s = blockIdx.x * blockDim.x + t;
  const int h = s < nseg ? segs[s].h : 0, J = s < nseg ? segs[s].J_hi : 0;
  pdl_wait();
  if (!CUT && nseg <= workers) {
    if (s < nseg) order[s] = s;
    return;
  }
  const int n = s >= nseg ? 0 : count ? count[s] : J + 1;
  int sum = 0;
  for (int i = t >> 7; i < num_heads; i += 2) sum += hist[i * kCountBuckets + (t & 127)];
  col[t >> 7][t & 127] = sum;
  __syncthreads();
  if (warp == 0) {   // scans over the classes, four per lane
    int c[4], u[4], x[4];
    float blocks = 0.f;
#pragma unroll
    for (int i = 0; i < 4; ++i) {
      c[i] = col[0][lane * 4 + i] + col[1][lane * 4 + i];
      blocks += (float)c[i] * (float)class_min_count(lane * 4 + i);
    }
#pragma unroll
    for (int o = 16; o > 0; o >>= 1) blocks += __shfl_xor_sync(0xffffffffu, blocks, o);
    const float share = blocks / (float)workers;
    int longest = 0;
#pragma unroll
    for (int i = 0; i < 4; ++i) longest = max(longest, c[i] > 0 ? class_min_count(lane * 4 + i) : 0);
    longest = CUT ? __reduce_max_sync(0xffffffffu, longest) : 0;
    const bool cutting = CUT && longest >= kCutMin && (float)longest > kCutFrom * share;
    int n_long = 0, n_cut = 0, long_classes = 0;
#pragma unroll
    for (int i = 0; i < 4; ++i) {
      const float len = (float)class_min_count(lane * 4 + i);
      const bool is_long = num_heads <= kMaxLongHeads && len * kLongShare > share;   // (holds for the first classes: they count down)
      if (is_long) {
        ++long_classes;
        n_long += c[i];
      } else {
        c[i] = 0;
      }
      u[i] = is_long && cutting && len >= (float)kCutMin ? min(kMaxCuts, max(1, (int)ceilf(len / (0.5f * share)))) : 1;
      x[i] = u[i] > 1 ? c[i] * u[i] : 0;
    }
    if (cutting) {
      const ClassScan slots(x, lane), segs_before(c, lane);   // (classes that are cut come before those that are not)
#pragma unroll
      for (int i = 0; i < 4; ++i) {
        if (slots.before[i] + x[i] > cut.max_slots) u[i] = 1;   // (a prefix: from the first class that does not fit, none is cut)
        n_cut += u[i] > 1 ? c[i] : 0;
        slots_before[lane * 4 + i] = slots.before[i];
        cuts_before[lane * 4 + i] = segs_before.before[i];
      }
    }
#pragma unroll
    for (int i = 0; i < 4; ++i) x[i] = c[i] * u[i];
    const ClassScan units(x, lane);
#pragma unroll
    for (int i = 0; i < 4; ++i) {
      before[lane * 4 + i] = units.before[i];
      if constexpr (CUT) parts[lane * 4 + i] = u[i];
    }
#pragma unroll
    for (int o = 16; o > 0; o >>= 1) {
      n_long += __shfl_xor_sync(0xffffffffu, n_long, o);
      n_cut += __shfl_xor_sync(0xffffffffu, n_cut, o);
      long_classes += __shfl_xor_sync(0xffffffffu, long_classes, o);
    }
    if (lane == 0) {
      s_num_long = units.total;
      s_first_short = long_classes;
      if (CUT && blockIdx.x == 0) {
        *cut.n_units = units.total + nseg - n_long;
        *cut.n_split = n_cut;
      }
    }
  }
  __syncthreads();
  const int first_short = s_first_short;
  for (int i = warp; first_short > 0 && i < num_heads; i += 8) {
    const int4 c = reinterpret_cast<const int4*>(hist + i * kCountBuckets)[lane];
    int x = (lane * 4 < first_short ? c.x : 0) + (lane * 4 + 1 < first_short ? c.y : 0) +
            (lane * 4 + 2 < first_short ? c.z : 0) + (lane * 4 + 3 < first_short ? c.w : 0);
#pragma unroll
    for (int o = 16; o > 0; o >>= 1) x += __shfl_xor_sync(0xffffffffu, x, o);
    if (lane == 0) head_long[i] = x;
  }
  __syncthreads();
  if (s >= nseg) return;
  const int b = order_bucket(h, n), cls = b - h * kCountBuckets;
  if (cls < first_short) {
    const int k = atomicAdd(&cursor[cls], 1), U = CUT ? parts[cls] : 1;   // (the cursors of head 0's long classes serve all heads)
    const int slot = U > 1 ? slots_before[cls] + k * U : 0;
    for (int u = 0; u < U; ++u) {
      order[before[cls] + k * U + u] = s;
      if constexpr (CUT) cut.unit_split[before[cls] + k * U + u] = pack_split(u, U, slot);
    }
    if (U > 1) {
      cut.seg_split[s] = pack_split(0, U, slot);
      cut.split_list[cuts_before[cls] + k] = s;
    }
    return;
  }
  int pos = s_num_long + h * per_head;
  for (int i = 0; first_short > 0 && i < h; ++i) pos -= head_long[i];
  const int32_t* row = hist + h * kCountBuckets;
#pragma unroll 4
  for (int i = first_short; i < cls; ++i) pos += row[i];
  pos += atomicAdd(&cursor[b], 1);
  order[pos] = s;
  if constexpr (CUT) cut.unit_split[pos] = pack_split(0, 1, 0);
}

// ----------------------------------------------------------------------------------------
// Pooled statistics carried from one chunk of a chunked prefill to the next (Sec. 4.3, "Compatibility with Chunked Prefill": the index stage runs once
// per chunk; without this every chunk pools the whole cached prefix again).  The means of a block that was
// complete in the previous chunk are the same numbers in this one: rows are copied from the previous workspace's
// layout to this plan's.  carry[3 b + {0, 1, 2}] = first source row, first destination row, rows to copy of
// sequence b.  grid (sequences, row groups of 8); a row of one array is Hkv x 128 elements.
// ----------------------------------------------------------------------------------------
__global__ void pool_carry_kernel(const int32_t* carry, int row_bytes16, int row_bytes8,
                                  const uint8_t* s_khi, const uint8_t* s_klo,
                                  const uint8_t* s_vbar, const uint8_t* s_k8hi,
                                  const uint8_t* s_k8lo, uint8_t* __restrict__ d_khi,
                                  uint8_t* __restrict__ d_klo, uint8_t* __restrict__ d_vbar,
                                  uint8_t* __restrict__ d_k8hi, uint8_t* __restrict__ d_k8lo) {
  pdl_trigger();
  pdl_wait();
  const int b = blockIdx.x;
  const int src0 = carry[3 * b], dst0 = carry[3 * b + 1], n = carry[3 * b + 2];
  for (int j = blockIdx.y * 8; j < n; j += gridDim.y * 8) {
    const int rows = min(8, n - j);
    auto copy = [&](const uint8_t* s, uint8_t* d, int rb) {
      if (rb == 0) return;
      const uint4* sp = reinterpret_cast<const uint4*>(s + (size_t)(src0 + j) * rb);
      uint4* dp = reinterpret_cast<uint4*>(d + (size_t)(dst0 + j) * rb);
      for (int i = threadIdx.x; i < rows * rb / 16; i += blockDim.x) dp[i] = sp[i];
    };
    copy(s_khi, d_khi, row_bytes16);
    copy(s_klo, d_klo, row_bytes16);
    copy(s_vbar, d_vbar, row_bytes16);
    copy(s_k8hi, d_k8hi, row_bytes8);
    copy(s_k8lo, d_k8lo, row_bytes8);
  }
}

}  // namespace fp2
