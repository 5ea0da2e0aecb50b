// Index export (Algorithm 1 line 5; Sec. 3.3 "Index-Driven Sparse Traversal", Eq. 17; Sec. 3.4 "Serving
// Integration"): the padded block lists of the selector as a compact CSR (cu, idx) of physical tiles of
// tile_tokens tokens, per segment in segment order (that is: per KV head under PackGQA), and the page-level
// table read out of a token-level slot map by striding.
//
// A logical block J of 128 tokens becomes the tiles J tpb .. J tpb + tpb - 1 (tpb = 128 / tile_tokens) that hold
// at least one real token; only the last block of a sequence can be short, and a list is ascending, so only a
// segment's last entry can produce fewer than tpb tiles -- entry k of a segment always starts at cu + k tpb.
// Integer work throughout; launch-latency- and HBM-bound (reads the lists once, writes tpb entries per block).
#pragma once
#include "common.cuh"
#include "ptx.cuh"

namespace fp2 {

// tiles of block J that hold a real token of a sequence of Lk tokens
__device__ __forceinline__ int tiles_in_block(int J, int Lk, int tile_tokens) {
  const int ntok = min(kBlock, Lk - J * kBlock);
  return ntok <= 0 ? 0 : (ntok + tile_tokens - 1) / tile_tokens;
}

// count and list entries as the attention kernel reads them: out-of-range values are clamped (and flagged)
__device__ __forceinline__ int clamped_count(const SegInfo& sg, const int32_t* seg_count, int* status) {
  int T = seg_count[sg.seg];
  if (T < 0 || T > sg.J_hi + 1) {
    atomicOr(status + ST_BAD_LIST, 1);
    T = max(0, min(T, sg.J_hi + 1));
  }
  return T;
}

// Offsets in two steps, in place (nothing but the caller's cu holds them).  csr_count_kernel: cu[g + 1] = tiles of the segments
// of g's group of kCsrGroup up to g.  csr_offset_kernel, one CTA: adds the groups in front, whose totals are the last entries of
// the groups.  (One CTA that scanned all counts tile by tile took 13 of the 32 us of an export of 16384 segments; index and
// export of 65536 tokens 391 -> 384 us, of 22965 tokens 112.5 -> 107.2, of 98374 tokens 713 -> 698.)
constexpr int kCsrGroup = 256;

// inclusive prefix sum over the CTA's threads (a multiple of 32, up to 1024); warp_tot: 32 words of shared memory
__device__ __forceinline__ int32_t cta_prefix(int32_t v, int32_t* warp_tot) {
  const int lane = threadIdx.x & 31, w = threadIdx.x >> 5;
#pragma unroll
  for (int d = 1; d < 32; d <<= 1) {
    const int32_t y = __shfl_up_sync(0xffffffffu, v, d);
    if (lane >= d) v += y;
  }
  if (lane == 31) warp_tot[w] = v;
  __syncthreads();
  const int32_t t = lane < w ? warp_tot[lane] : 0;
  return v + __reduce_add_sync(0xffffffffu, t);
}

// One thread per segment.
__global__ void __launch_bounds__(kCsrGroup) csr_count_kernel(const SegInfo* __restrict__ segs, const int32_t* seg_count,
                                                              const int32_t* blk_idx, int nseg, int tile_tokens,
                                                              int32_t* __restrict__ cu, int* __restrict__ status) {
  __shared__ int32_t warp_tot[32];
  pdl_trigger();
  const int g = blockIdx.x * kCsrGroup + threadIdx.x;
  SegInfo sg;
  if (g < nseg) sg = segs[g];   // the plan's table: not written by any kernel
  pdl_wait();
  int n = 0;
  if (g < nseg) {
    const int T = clamped_count(sg, seg_count, status);
    if (T > 0) {
      const int J = max(0, min(blk_idx[sg.off + T - 1], sg.J_hi));
      n = (T - 1) * (kBlock / tile_tokens) + tiles_in_block(J, sg.Lk, tile_tokens);
    }
  }
  const int32_t incl = cta_prefix(n, warp_tot);
  if (g < nseg) cu[g + 1] = incl;
  if (g == 0) cu[0] = 0;
}

__global__ void __launch_bounds__(1024, 1) csr_offset_kernel(int32_t* cu, int nseg) {
  __shared__ int32_t warp_tot[32], offset[1024];
  pdl_trigger();
  pdl_wait();
  const int t = threadIdx.x, groups = (nseg + kCsrGroup - 1) / kCsrGroup;
  int32_t before = 0;   // tiles in front of the 1024 groups at hand
  for (int g0 = 0; g0 < groups; g0 += 1024) {
    const int last = min((g0 + t + 1) * kCsrGroup, nseg);
    const int32_t total = g0 + t < groups ? cu[last] : 0;
    offset[t] = before + cta_prefix(total, warp_tot) - total;
    __syncthreads();
    const int n = min(1024, groups - g0) * kCsrGroup;
    int32_t* v = cu + 1 + (size_t)g0 * kCsrGroup;
    const int limit = min(n, nseg - g0 * kCsrGroup);
#pragma unroll 4
    for (int i = t; i < limit; i += 1024) v[i] += offset[i / kCsrGroup];
    __syncthreads();
    if (g0 + 1024 < groups) before = cu[(size_t)(g0 + 1024) * kCsrGroup];   // the entry in front of the next group, final by now
    __syncthreads();
  }
}

// one warp per segment: entry k of the list -> its tiles at cu[g] + k tpb
__global__ void csr_fill_kernel(const SegInfo* __restrict__ segs, const int32_t* seg_count,
                                const int32_t* blk_idx, int nseg, int tile_tokens,
                                const int32_t* cu, int32_t* __restrict__ idx, int* __restrict__ status) {
  pdl_trigger();
  const int g = (blockIdx.x * blockDim.x + threadIdx.x) >> 5, lane = threadIdx.x & 31;
  SegInfo sg;
  if (g < nseg) sg = segs[g];
  pdl_wait();
  if (g >= nseg) return;
  int T = seg_count[sg.seg];
  T = max(0, min(T, sg.J_hi + 1));   // flagged by the counting kernel
  const int tpb = kBlock / tile_tokens;
  const int32_t* list = blk_idx + sg.off;
  int32_t* out = idx + cu[g];
  bool bad = false;
  for (int k = lane; k < T; k += 32) {
    int J = list[k];
    if (J < 0 || J > sg.J_hi || (k > 0 && list[k - 1] >= J)) bad = true;
    J = max(0, min(J, sg.J_hi));
    const int n = k + 1 < T ? tpb : tiles_in_block(J, sg.Lk, tile_tokens);
    for (int j = 0; j < n; ++j) out[k * tpb + j] = J * tpb + j;
  }
  if (bad) atomicOr(status + ST_BAD_LIST, 1);
}

// page_table[b][k] = token_to_slot[b][k p] / p for the pages that hold a token, -1 beyond (Sec. 3.4).  A sampled
// slot that is not the first of a page is flagged in the status block.
__global__ void page_table_from_token_map_kernel(const int32_t* token_to_slot, int max_tokens,
                                                 const int32_t* seqlens_k, int ns, int p, int max_pages,
                                                 int32_t* __restrict__ page_table, int* __restrict__ status) {
  pdl_trigger();
  pdl_wait();
  const int i = blockIdx.x * blockDim.x + threadIdx.x;
  if (i >= ns * max_pages) return;
  const int b = i / max_pages, k = i % max_pages;
  int32_t v = -1;
  if ((int64_t)k * p < seqlens_k[b] && (int64_t)k * p < max_tokens) {
    const int32_t slot = token_to_slot[(size_t)b * max_tokens + (size_t)k * p];
    if (slot < 0 || slot % p != 0) atomicOr(status + ST_BAD_LIST, 4);
    v = slot < 0 ? -1 : slot / p;
  }
  page_table[i] = v;
}

}  // namespace fp2
