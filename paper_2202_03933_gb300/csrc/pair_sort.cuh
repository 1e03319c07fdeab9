// Order in which the pair kernels take their pairs: batches sorted by cost, so
// that the lanes of a warp run pairs of the same kind.
#pragma once

#include "clip.cuh"
#include "context.h"
#include "quadrature.cuh"

namespace mortar {

namespace {

// Shared memory of a warp with batches of B pairs: the set of key values
// present, the sorted order and the sort keys of its batch.
__host__ __device__ constexpr int batch_smem_bytes(int B) { return 8 * 4 + B * 3; }

// Guided self-scheduling: a warp takes half an even share of the pairs left
// (at most B, at least 32, a multiple of 32); false when none are left.
// share: twice the number of warps.
__device__ __forceinline__ bool fetch_batch(unsigned long long* work_ctr, int64_t n, int64_t share, int B,
                                            int64_t& base, int& fetch) {
  base = 0;
  fetch = B;
  if ((threadIdx.x & 31) == 0) {
    const unsigned long long seen = *reinterpret_cast<volatile unsigned long long*>(work_ctr);
    const int64_t f = (n - (int64_t)seen) / share;
    fetch = f >= B ? B : (f < 32 ? 32 : (int)(f & ~31ll));
    base = (int64_t)atomicAdd(work_ctr, (unsigned long long)fetch);
  }
  base = __shfl_sync(0xffffffffu, base, 0);
  fetch = __shfl_sync(0xffffffffu, fetch, 0);
  return base < n;
}

// Sorts the batch [base, lim) by a cost key, descending, into the order at
// my + 32 (uint16, relative to base); returns its length.  Key: 1 + 16 x the
// cell count + the edge intersections of an FP32 clip (0 = no pair); a cost
// estimate only, the FP64 clip decides.  Counting sort over the key values
// present, by ballots.  my: the warp's batch memory (batch_smem_bytes(B)).
// SUB: units per pair (4 for quadratic slave elements: unit u is sub-element
// u % 4 of pair u / 4, with a record of its own).
template <int NS, int NM, int SUB>
__device__ __forceinline__ int sort_batch(unsigned char* my, int B, int64_t base, int64_t lim, int rounds,
                                          const int32_t* __restrict__ ps, const int32_t* __restrict__ pm,
                                          const double* __restrict__ srec, const double* __restrict__ xm,
                                          const int32_t* __restrict__ conn_m) {
  unsigned* pres = reinterpret_cast<unsigned*>(my);
  uint16_t* perm = reinterpret_cast<uint16_t*>(my + 32);
  uint8_t* keys = reinterpret_cast<uint8_t*>(perm + B);
  const int lane = threadIdx.x & 31;
  const unsigned lt_mask = (1u << lane) - 1u;
  if (lane < 8) pres[lane] = 0u;
  __syncwarp();
#pragma unroll 1
  for (int rr = 0; rr < rounds; ++rr) {
    const int64_t p = base + rr * 32 + lane;
    int key = 0;
    if (p < lim) {
      int n_int = 0;
      const int64_t pair = p / SUB;
      const double* r = srec + (int64_t)SR_STRIDE * (SUB * (int64_t)ps[pair] + p % SUB);
      const int nr = clip_count_f32<NS, NM>(r, xm, conn_m, pm[pair], n_int);
      key = 1 + 16 * (nr == 0 ? 0 : (nr == 3 ? 1 : min(nr, kPolyS))) + min(n_int, 15);
      atomicOr(&pres[key >> 5], 1u << (key & 31));
    }
    keys[rr * 32 + lane] = (uint8_t)key;
  }
  __syncwarp();
  int basecnt = 0;
#pragma unroll 1
  for (int w = 7; w >= 0; --w) {
    unsigned bits = pres[w];
    while (bits != 0u) {   // uniform across the warp
      const int b = 31 - __clz(bits);
      bits &= ~(1u << b);
      const int v = 32 * w + b;
      int before = 0;
#pragma unroll 1
      for (int rr = 0; rr < rounds; ++rr) {
        const int slot = rr * 32 + lane;
        const bool hit = keys[slot] == v;
        const unsigned mk = __ballot_sync(0xffffffffu, hit);
        if (hit) perm[basecnt + before + __popc(mk & lt_mask)] = (uint16_t)slot;
        before += __popc(mk);
      }
      basecnt += before;
    }
  }
  __syncwarp();
  return basecnt;
}

// Writes the sorted order of every batch of the chunk that begins at pair
// `first`: order[base + i] = pair, relative to it.  A kernel of
// its own, so that the pair kernels' code stays within the instruction cache,
// and because it is latency-bound where they are not: small batches' worth of
// registers, many warps.
constexpr int kSortThreads = 128;
// Forward pair kernels at 600x520 with batches of 64, 256 and 1024 pairs: 3.02, 2.98,
// 2.99 ms; the sort itself takes 0.20 ms.
constexpr int kSortBatch = 1024;   // default pairs per warp batch, and the most
template <int NS, int NM, int SUB>
__global__ void __launch_bounds__(kSortThreads) k_pair_sort(
    const int32_t* __restrict__ ps, const int32_t* __restrict__ pm, const double* __restrict__ srec,
    const double* __restrict__ xm, const int32_t* __restrict__ conn_m, int64_t pair_cap, int64_t first, int B,
    int32_t watchdog_us,
    int32_t* __restrict__ order, DevStatus* st) {
  extern __shared__ __align__(16) unsigned char smem_raw[];
  unsigned char* my = smem_raw + (size_t)(threadIdx.x >> 5) * batch_smem_bytes(B);
  const uint16_t* perm = reinterpret_cast<const uint16_t*>(my + 32);
  const int64_t n = SUB * chunk_pairs(st, pair_cap, first, kPairChunk / SUB);   // units
  ps += first;
  pm += first;
  const int64_t share = 2 * (int64_t)gridDim.x * (blockDim.x >> 5);
  const Watchdog wd(watchdog_us);
  for (;;) {   // bounded: the shared counter only grows
    if (wd.expired(&st->timeout)) break;
    int64_t base;
    int fetch;
    if (!fetch_batch(&st->pair_ctr[0], n, share, B, base, fetch)) break;
    const int64_t lim = min(n, base + (int64_t)fetch);
    const int live = sort_batch<NS, NM, SUB>(my, B, base, lim, (fetch + 31) >> 5, ps, pm, srec, xm, conn_m);
    for (int i = threadIdx.x & 31; i < live; i += 32) order[base + i] = (int32_t)(base + perm[i]);
    __syncwarp();
  }
}

template <int NS, int NM, int SUB = 1>
void launch_pair_sort(const IntegrateArgs& a, const RunParams& rp, int n_sm, int B, int64_t first) {
  cudaMemsetAsync(&a.st->pair_ctr, 0, sizeof(a.st->pair_ctr), a.stream);   // the chunk's kernels
  auto kern = k_pair_sort<NS, NM, SUB>;
  const size_t shm = (size_t)(kSortThreads / 32) * batch_smem_bytes(B);
  int per_sm = 0;
  cudaOccupancyMaxActiveBlocksPerMultiprocessor(&per_sm, kern, kSortThreads, shm);
  kern<<<(unsigned)(n_sm * (per_sm < 1 ? 1 : per_sm)), kSortThreads, shm, a.stream>>>(
      a.ps, a.pm, a.srec, a.xm, a.conn_m, a.pair_cap, first, B, rp.watchdog_us, a.order, a.st);
}

}  // namespace

}  // namespace mortar
