// lookback.cuh -- prefixes over the tiles of one launch by decoupled look-back
// (Merrill & Garland): a tile publishes its own count at once and its inclusive
// prefix when it knows it; a reader adds the counts of the tiles before it
// until it meets a prefix.  Tiles are numbered by a counter as blocks start, so
// every tile that a block waits for is already running; the waits are bounded
// all the same, and one that runs out sets SPH_ST_TIMEOUT and is passed on as a
// failure to the tiles behind it.
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
  static constexpr W kFailed = (W)3 << kShift;  // a wait ran out
  static constexpr W kValue = kCount - 1;
};
constexpr int kPollLimit = 1 << 22;  // polls of one wait (seconds)

template <class W>
__device__ __forceinline__ W pub_load(const W* p) {
  return *(const volatile W*)p;
}
template <class W>
__device__ __forceinline__ void pub_store(W* p, W v) {
  *(volatile W*)p = v;
}
template <class W>
__device__ __forceinline__ bool pub_is_last(W v) {  // a prefix, or a failure
  return (v & Pub<W>::kPrefix) != 0;
}
template <class W>
__device__ __forceinline__ bool pub_is_failed(W v) {
  return (v & Pub<W>::kFailed) == Pub<W>::kFailed;
}

template <class W>
__device__ __forceinline__ W pub_wait(const W* p) {
  W v = pub_load(p);
  for (int it = 0; v == 0 && it < kPollLimit; ++it) {
    if (it > 8) __nanosleep(40);
    v = pub_load(p);
  }
  return v != 0 ? v : Pub<W>::kFailed;
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

// Publishes tile's count tot and finds the sum of the tiles before it, into
// *before (-1 if a wait ran out).  Called by the block's first warp; 32 tiles
// back at a time.
__device__ __forceinline__ void lookback(uint64_t* pub, int32_t tile, int32_t tot, int32_t* before, int32_t* status) {
  using P = Pub<uint64_t>;
  const int lane = threadIdx.x & 31;
  if (lane == 0) pub_store(pub + tile, (tile == 0 ? P::kPrefix : P::kCount) | (uint64_t)tot);
  int32_t sum = 0;
  bool failed = false;
  for (int32_t t = tile - 1 - lane; tile > 0; t -= 32) {
    const uint64_t w = t >= 0 ? pub_wait(pub + t) : P::kPrefix;
    const unsigned last = __ballot_sync(0xffffffffu, pub_is_last(w));
    const bool use = last == 0u || lane < __ffs((int)last);
    failed = __any_sync(0xffffffffu, use && pub_is_failed(w));
    int32_t x = use ? (int32_t)(w & P::kValue) : 0;
#pragma unroll
    for (int o = 16; o > 0; o >>= 1) x += __shfl_xor_sync(0xffffffffu, x, o);
    sum += x;
    if (last != 0u || failed) break;
  }
  if (lane == 0) {
    if (tile > 0) pub_store(pub + tile, failed ? P::kFailed : P::kPrefix | (uint64_t)(sum + tot));
    if (failed) atomicOr(status, SPH_ST_TIMEOUT);
    *before = failed ? -1 : sum;
  }
}

}  // namespace sphk
