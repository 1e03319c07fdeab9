// Ragged output in one visit.  A counting kernel whose blocks own 128
// consecutive rows (or slave elements) each, and whose threads hold their row
// when they have counted it, leaves the rows in a staging area instead of
// dropping them: a block takes room for all of its rows from a counter and
// notes where.  When the counts have been scanned into offsets, the block's
// rows are contiguous in the output too, and the writing kernel only copies.
// A block that found no room, or has a row too long to be held, is not staged
// (kNotStaged); its rows are visited again by the writing kernel.
#pragma once

#include "context.h"

namespace mortar {

constexpr long long kNotStaged = -1;

// The area: one position per block, then the entries.
struct Staging {
  long long* base;             // of each block
  char* data;
  int64_t bytes;               // of data
  unsigned long long* taken;   // counter, entries
};

// memory: the clip records' workspace, which is idle before and after the pair kernels.
inline Staging staging_area(const DevBuf& b, int64_t blocks, unsigned long long* taken) {
  const int64_t head = (8 * blocks + 255) / 256 * 256;
  char* p = static_cast<char*>(b.p);
  if (!p || (int64_t)b.bytes < head + 4096) return {nullptr, nullptr, 0, taken};
  return {reinterpret_cast<long long*>(p), p + head, (int64_t)b.bytes - head, taken};
}

// Position of this thread's `mine` of its block's entries among the block's, and
// the block's total; every thread of the block (at most 1024) calls it.
__device__ __forceinline__ unsigned block_exclusive(unsigned mine, unsigned& total) {
  __shared__ unsigned warp_sum[32];
  const int lane = threadIdx.x & 31, warp = threadIdx.x >> 5;
  unsigned v = mine;
#pragma unroll
  for (int d = 1; d < 32; d <<= 1) {
    const unsigned w = __shfl_up_sync(0xffffffffu, v, d);
    if (lane >= d) v += w;
  }
  if (lane == 31) warp_sum[warp] = v;
  __syncthreads();
  unsigned before = 0;
  total = 0;
  for (int w = 0; w < (int)((blockDim.x + 31) >> 5); ++w) {
    if (w < warp) before += warp_sum[w];
    total += warp_sum[w];
  }
  return before + v - mine;
}

// Room for n entries of this block (size bytes each), kNotStaged if there is
// none or !fits; noted for the writing kernel.  Every thread calls it.
__device__ __forceinline__ long long stage_block(const Staging& s, bool fits, int64_t n, int64_t size) {
  __shared__ long long at;
  if (threadIdx.x == 0) {
    at = kNotStaged;
    if (s.base) {
      if (fits) {
        at = (long long)atomicAdd(s.taken, (unsigned long long)n);
        if ((at + n) * size > s.bytes) at = kNotStaged;
      }
      s.base[blockIdx.x] = at;
    }
  }
  __syncthreads();
  return at;
}

}  // namespace mortar
