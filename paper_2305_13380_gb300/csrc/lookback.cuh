// lookback.cuh -- prefixes over the tiles of one launch by decoupled look-back
// (Merrill & Garland): a tile publishes its own count at once and its inclusive
// prefix when it knows it; a reader adds the counts of the tiles before it
// until it meets a prefix.  Tiles are numbered by a counter as blocks start, so
// every tile that a block waits for is already running; the waits are bounded
// all the same, and a block whose wait runs out counts the items of all tiles
// before its own itself (the inputs are not written while a launch reads them):
// slower, the same prefix.
#pragma once
#include "sph_internal.cuh"

namespace sphk {

constexpr int kScanThreads = 256;
constexpr int kScanWarps = kScanThreads / 32;

// A published word: a value and, in the top two bits, its state (0: not yet).  The
// sort's are of 32 bits, a digit's items (the library takes fewer than 2^27); the
// scans' of 64, sums up to 2^31 - 1.
template <class W>
struct Pub {
  static constexpr int kShift = 8 * (int)sizeof(W) - 2;
  static constexpr W kCount = (W)1 << kShift;   // the tile's own count
  static constexpr W kPrefix = (W)2 << kShift;  // the inclusive prefix up to the tile
  static constexpr W kValue = kCount - 1;
};
// Polls of one wait (seconds).  -1: no published word is ever seen, every tile
// counts for itself (the tests build that).
#ifndef SPH_POLL_LIMIT
#define SPH_POLL_LIMIT (1 << 22)
#endif
constexpr int kPollLimit = SPH_POLL_LIMIT;

template <class W>
__device__ __forceinline__ W pub_load(const W* p) {
  return kPollLimit < 0 ? (W)0 : *(const volatile W*)p;
}
template <class W>
__device__ __forceinline__ void pub_store(W* p, W v) {
  *(volatile W*)p = v;
}
template <class W>
__device__ __forceinline__ bool pub_is_prefix(W v) {
  return (v & Pub<W>::kPrefix) != 0;
}

// The word, or 0 if the wait ran out.
template <class W>
__device__ __forceinline__ W pub_wait(const W* p) {
  W v = pub_load(p);
  for (int it = 0; v == 0 && it < kPollLimit; ++it) {
    if (it > 8) __nanosleep(40);
    v = pub_load(p);
  }
  return v;
}

// Exclusive scan of one value per thread over a block of kScanThreads; total in
// *total.
__device__ __forceinline__ int32_t block_scan(int32_t v, int32_t* total) {
  __shared__ int32_t ws[kScanWarps];
  const int lane = threadIdx.x & 31, w = threadIdx.x >> 5;
  int32_t x = v;
#pragma unroll
  for (int o = 1; o < 32; o <<= 1) {
    const int32_t t = __shfl_up_sync(0xffffffffu, x, o);
    if (lane >= o) x += t;
  }
  if (lane == 31) ws[w] = x;
  __syncthreads();
  int32_t wbase = 0, tot = 0;
#pragma unroll
  for (int k = 0; k < kScanWarps; ++k) {
    wbase += k < w ? ws[k] : 0;
    tot += ws[k];
  }
  __syncthreads();
  *total = tot;
  return wbase + x - v;
}

// Publishes tile's count tot and finds the sum of the tiles before it.  Called by
// the block's first warp; 32 tiles back at a time.  -1 if a wait ran out.
__device__ __forceinline__ int32_t lookback(uint64_t* pub, int32_t tile, int32_t tot) {
  using P = Pub<uint64_t>;
  const int lane = threadIdx.x & 31;
  if (lane == 0) pub_store(pub + tile, (tile == 0 ? P::kPrefix : P::kCount) | (uint64_t)tot);
  int32_t sum = 0;
  for (int32_t t = tile - 1 - lane; tile > 0; t -= 32) {
    const uint64_t w = t >= 0 ? pub_wait(pub + t) : P::kPrefix;
    const unsigned last = __ballot_sync(0xffffffffu, pub_is_prefix(w));
    const bool use = last == 0u || lane < __ffs((int)last);
    if (__any_sync(0xffffffffu, use && w == 0)) return -1;
    int32_t x = use ? (int32_t)(w & P::kValue) : 0;
#pragma unroll
    for (int o = 16; o > 0; o >>= 1) x += __shfl_xor_sync(0xffffffffu, x, o);
    sum += x;
    if (last != 0u) break;
  }
  if (lane == 0 && tile > 0) pub_store(pub + tile, P::kPrefix | (uint64_t)(sum + tot));
  return sum;
}

// The sum of the tiles before tile, of `items` items in all, for every thread of
// the block: by look-back, or counted (count(i): item i's) where a wait ran out.
// (*s_before is free again after the caller's next barrier.)
template <class Count>
__device__ __forceinline__ int32_t tiles_before(uint64_t* pub, int32_t tile, int32_t tot, int64_t items,
                                                int32_t* s_before, Count count) {
  if (threadIdx.x < 32) {
    const int32_t b = lookback(pub, tile, tot);
    if (threadIdx.x == 0) *s_before = b;
  }
  __syncthreads();
  const int32_t before = *s_before;
  if (before >= 0) return before;
  int32_t mine = 0, all;
#pragma unroll 1
  for (int64_t i = threadIdx.x; i < items; i += kScanThreads) mine += count(i);
  block_scan(mine, &all);
  if (threadIdx.x == 0) pub_store(pub + tile, Pub<uint64_t>::kPrefix | (uint64_t)(all + tot));
  return all;
}

}  // namespace sphk
