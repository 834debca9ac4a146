// radix.cu -- stable least-significant-digit radix sort of (key, index) and
// exclusive scans, one pass over memory each.  Indices enter in ascending
// order, so equal keys keep ascending index: the result is exactly the stable
// counting sort of the cell grid (Sec. 2.1), for any cell size.
//
//   k_radix_hist  the digit counts of every pass, from one read of the keys
//   k_radix_pass  one 8-bit digit: a tile of 2048 items ranks its keys (equal
//                 digits within a warp + running per-warp counts), finds by
//                 look-back how many equal digits the tiles before it hold
//                 (lookback.cuh, a word per tile and digit), and writes the tile
//                 in order of digits, equal ones as one run.  A pass whose keys
//                 all share the digit (the bits beyond the cells in use) only
//                 copies.
//   k_radix_small all passes of up to 8192 items in one block
//   k_scan        exclusive scan, tiles of 4096, the same look-back
//
// They are bound by the latency of the look-back, not by bandwidth.  Seven passes
// over 2M 64-bit keys take 203 us (277 with every item scattered by itself: its
// sector of 32 bytes for 8; 343 as a histogram, three scan kernels and a
// scatter).  6,000 keys, six passes: 58 us with the histogram as launches, 36 in
// one block, which is bound by its one SM.
//
// A tile whose wait ran out counts the digits before it itself (lookback.cuh): the
// same order.
#include "lookback.cuh"
#include "per_device.h"
#include "sph_internal.cuh"
#include "sph_launch.h"

namespace sphk {

constexpr int kRadixItems = 8;
constexpr int kRadixTile = kScanThreads * kRadixItems;
constexpr int kRadixMaxPasses = 8;

// Digit counts of `passes` 8-bit digits of n keys, added to hist[pass * 256 + d].
template <class K>
__global__ void k_radix_hist(int64_t n, const K* __restrict__ keys, int passes, int32_t* __restrict__ hist) {
  __shared__ int32_t h[kRadixMaxPasses * 256];
  for (int i = threadIdx.x; i < passes * 256; i += kScanThreads) h[i] = 0;
  __syncthreads();
  const int lane = threadIdx.x & 31;
  for (int64_t base = (int64_t)blockIdx.x * kRadixTile; base < n; base += (int64_t)gridDim.x * kRadixTile) {
    K key[kRadixItems];
#pragma unroll
    for (int i = 0; i < kRadixItems; ++i) {
      const int64_t p = base + i * kScanThreads + threadIdx.x;
      key[i] = p < n ? keys[p] : (K)0;
    }
#pragma unroll
    for (int i = 0; i < kRadixItems; ++i) {
      const int64_t p0 = base + i * kScanThreads + (threadIdx.x & ~31);
      const bool ok = p0 + lane < n;
      for (int s = 0; s < passes; ++s) {
        const int d = (int)((key[i] >> (8 * s)) & 255);
        // the leading digits mostly agree within a warp: one add for all
        if (p0 + 31 < n && __all_sync(0xffffffffu, d == __shfl_sync(0xffffffffu, d, 0))) {
          if (lane == 0) atomicAdd(&h[s * 256 + d], 32);
        } else if (ok) {
          atomicAdd(&h[s * 256 + d], 1);
        }
      }
    }
  }
  __syncthreads();
  for (int i = threadIdx.x; i < passes * 256; i += kScanThreads)
    if (h[i] != 0) atomicAdd(&hist[i], h[i]);
}

// The lanes with ok and the digit d of this one.  A match costs as much as there
// are distinct digits in the warp: few in cell indices and levels, where
// neighbours in memory are mostly neighbours in space, up to 32 in the low bits
// of 64-bit Morton keys, where eight ballots are cheaper (seven passes over 2M
// keys: 230 -> 203 us; four over 2M cell indices: 89 -> 96 us).
template <class K>
__device__ __forceinline__ unsigned digit_peers(int d, bool ok) {
  if constexpr (sizeof(K) < 8) {
    return __match_any_sync(0xffffffffu, ok ? d : 256 + (int)(threadIdx.x & 31));  // !ok: no peers
  } else {
    unsigned peers = __ballot_sync(0xffffffffu, ok);
#pragma unroll
    for (int b = 0; b < 8; ++b) {
      const bool one = (d >> b) & 1;
      const unsigned m = __ballot_sync(0xffffffffu, one);
      peers &= one ? m : ~m;
    }
    return peers;
  }
}

// One pass.  Warp w of a tile handles items base + w * 256 + j * 32 + lane,
// j = 0..7, i.e. 8 consecutive groups of 32 consecutive items: processing j in
// order visits the warp's items in index order.  vals_in null: the values are
// the indices.  keys_out null: the keys are not needed any more.
template <class K>
__global__ void __launch_bounds__(kScanThreads)
k_radix_pass(int64_t n, const K* __restrict__ keys_in, const int32_t* __restrict__ vals_in, int shift,
             const int32_t* __restrict__ hist, int32_t* __restrict__ ticket, uint32_t* pub, K* __restrict__ keys_out,
             int32_t* __restrict__ vals_out) {
  __shared__ int32_t wcount[kScanWarps][256];
  __shared__ int32_t first[256];  // place of digit d's item i of the ordered tile: first[d] + i
  __shared__ K skeys[kRadixTile];
  __shared__ int32_t svals[kRadixTile];
  __shared__ int32_t s_tile;
  using Word = Pub<uint32_t>;
  const int warp = threadIdx.x >> 5, lane = threadIdx.x & 31, d0 = threadIdx.x;
  const int32_t all = hist[d0];
  if (d0 == 0) s_tile = atomicAdd(ticket, 1);
  for (int d = lane; d < 256; d += 32) wcount[warp][d] = 0;
  const bool same = __syncthreads_or((int64_t)all == n);
  const int32_t tile = s_tile;
  const int64_t base = (int64_t)tile * kRadixTile + warp * (32 * kRadixItems);
  K key[kRadixItems];
  int32_t val[kRadixItems], rank[kRadixItems];
#pragma unroll
  for (int j = 0; j < kRadixItems; ++j) {
    const int64_t p = base + j * 32 + lane;
    key[j] = p < n ? keys_in[p] : (K)0;
    val[j] = p < n ? (vals_in != nullptr ? vals_in[p] : (int32_t)p) : 0;
  }
  if (!same) {  // (else every key has this digit)
    int32_t tot_all;
    const int32_t dst0 = block_scan(all, &tot_all);  // first place of digit d0
    const unsigned lt = (1u << lane) - 1u;
#pragma unroll
    for (int j = 0; j < kRadixItems; ++j) {
      const bool ok = base + j * 32 + lane < n;
      const int d = (int)((key[j] >> shift) & 255);
      const unsigned peers = digit_peers<K>(d, ok);
      int r = 0;
      if (ok) r = wcount[warp][d] + __popc(peers & lt);
      rank[j] = r;
      __syncwarp();
      // the highest lane of each group of equal digits advances the count
      if (ok && (peers >> lane) == 1u) wcount[warp][d] += __popc(peers);
      __syncwarp();
    }
    __syncthreads();
    // the tile's count of digit d0, and each warp's first place within the tile
    int32_t mine = 0;
#pragma unroll
    for (int w = 0; w < kScanWarps; ++w) {
      const int32_t c = wcount[w][d0];
      wcount[w][d0] = mine;
      mine += c;
    }
    uint32_t* my = pub + (int64_t)tile * 256 + d0;
    pub_store(my, (tile == 0 ? Word::kPrefix : Word::kCount) | (uint32_t)mine);
    // the tile in order of digits, in shared memory
    int32_t cnt;
    const int32_t at0 = block_scan(mine, &cnt);
#pragma unroll
    for (int w = 0; w < kScanWarps; ++w) wcount[w][d0] += at0;
    __syncthreads();
#pragma unroll
    for (int j = 0; j < kRadixItems; ++j) {
      if (base + j * 32 + lane < n) {
        const int at = wcount[warp][(int)((key[j] >> shift) & 255)] + rank[j];
        skeys[at] = key[j];
        svals[at] = val[j];
      }
    }
    int32_t before = 0;
    bool expired = false;
    for (int32_t t = tile - 1; t >= 0;) {
      // four tiles back at a time, their words in flight together (eight: 230 us for
      // the seven passes over 2M keys instead of 208, sixteen: 242)
      uint32_t v[4];
#pragma unroll
      for (int i = 0; i < 4; ++i) v[i] = t - i >= 0 ? pub_load(pub + (int64_t)(t - i) * 256 + d0) : Word::kPrefix;
      bool stop = false;
#pragma unroll
      for (int i = 0; i < 4; ++i) {
        if (!stop && t - i >= 0) {
          if (v[i] == 0u) v[i] = pub_wait(pub + (int64_t)(t - i) * 256 + d0);
          expired = v[i] == 0u;
          stop = expired || pub_is_prefix(v[i]);
          before += (int32_t)(v[i] & Word::kValue);
        }
      }
      if (stop) break;
      t -= 4;
    }
    if (tile > 0 && !expired) pub_store(my, Word::kPrefix | (uint32_t)(before + mine));
    first[d0] = dst0 + before - at0;
    if (__syncthreads_or(expired)) {
      wcount[0][d0] = 0;
      __syncthreads();
#pragma unroll 1
      for (int64_t p = d0; p < (int64_t)tile * kRadixTile; p += kScanThreads)
        atomicAdd(&wcount[0][(int)((keys_in[p] >> shift) & 255)], 1);
      __syncthreads();
      before = wcount[0][d0];
      pub_store(my, Word::kPrefix | (uint32_t)(before + mine));
      first[d0] = dst0 + before - at0;
      __syncthreads();
    }
    // equal digits leave as runs of consecutive places
#pragma unroll
    for (int j = 0; j < kRadixItems; ++j) {
      const int at = j * kScanThreads + d0;
      if (at < cnt) {
        const K k = skeys[at];
        const int64_t dst = (int64_t)first[(int)((k >> shift) & 255)] + at;
        if (keys_out != nullptr) keys_out[dst] = k;
        vals_out[dst] = svals[at];
      }
    }
    return;
  }
#pragma unroll
  for (int j = 0; j < kRadixItems; ++j) {
    const int64_t p = base + j * 32 + lane;
    if (p < n) {
      if (keys_out != nullptr) keys_out[p] = key[j];
      vals_out[p] = val[j];
    }
  }
}

// All passes of up to kSmallMax items in one block: the items of a warp (256
// consecutive ones) are ranked as in k_radix_pass, the whole of them reordered in
// shared memory, pass after pass.
constexpr int kSmallMax = 8192;
constexpr int kSmallItems = 8;
template <class K>
__host__ __device__ constexpr size_t small_smem() {
  return (size_t)kSmallMax * (sizeof(K) + sizeof(int32_t)) + (size_t)(kSmallMax / 256) * 256 * sizeof(uint16_t);
}

template <class K>
__global__ void __launch_bounds__(kSmallMax / kSmallItems)
k_radix_small(int n, const K* __restrict__ keys_in, int passes, K* __restrict__ keys_out,
              int32_t* __restrict__ vals_out) {
  extern __shared__ __align__(16) unsigned char rsm[];
  int32_t* svals = reinterpret_cast<int32_t*>(rsm + (size_t)kSmallMax * sizeof(K));
  K* skeys = reinterpret_cast<K*>(rsm);
  uint16_t* counts = reinterpret_cast<uint16_t*>(svals + kSmallMax);  // [warp][digit]
  __shared__ int32_t ws[8];
  const int t = threadIdx.x, warp = t >> 5, lane = t & 31, nw = blockDim.x >> 5;
  const int base = warp * (32 * kSmallItems);
  const unsigned lt = (1u << lane) - 1u;
  K key[kSmallItems];
  int32_t val[kSmallItems], rank[kSmallItems];
#pragma unroll
  for (int j = 0; j < kSmallItems; ++j) {
    const int p = base + j * 32 + lane;
    key[j] = p < n ? keys_in[p] : (K)0;
    val[j] = p;
  }
#pragma unroll 1
  for (int pass = 0; pass < passes; ++pass) {
    const int shift = 8 * pass;
    uint16_t* mine = counts + warp * 256;
    *reinterpret_cast<uint4*>(mine + 8 * lane) = make_uint4(0u, 0u, 0u, 0u);
    __syncwarp();
#pragma unroll
    for (int j = 0; j < kSmallItems; ++j) {
      const bool ok = base + j * 32 + lane < n;
      const int d = (int)((key[j] >> shift) & 255);
      const unsigned peers = digit_peers<K>(d, ok);
      int r = 0;
      if (ok) r = mine[d] + __popc(peers & lt);
      rank[j] = r;
      __syncwarp();
      if (ok && (peers >> lane) == 1u) mine[d] = (uint16_t)(mine[d] + __popc(peers));
      __syncwarp();
    }
    __syncthreads();
    // digit t: its items of the warps before each warp, and its first place
    int32_t sum = 0;
    if (t < 256) {
#pragma unroll 8
      for (int w = 0; w < nw; ++w) {
        const int32_t c = counts[w * 256 + t];
        counts[w * 256 + t] = (uint16_t)sum;
        sum += c;
      }
    }
    if (__syncthreads_or(t < 256 && sum == n)) continue;  // every key has this digit
    int32_t x = sum;
#pragma unroll
    for (int o = 1; o < 32; o <<= 1) {
      const int32_t v = __shfl_up_sync(0xffffffffu, x, o);
      if (lane >= o) x += v;
    }
    if (t < 256 && lane == 31) ws[warp] = x;
    __syncthreads();
    if (t < 256) {
      int32_t first = x - sum;
      for (int k = 0; k < warp; ++k) first += ws[k];
      for (int w = 0; w < nw; ++w) counts[w * 256 + t] = (uint16_t)(counts[w * 256 + t] + first);
    }
    __syncthreads();
#pragma unroll
    for (int j = 0; j < kSmallItems; ++j) {
      if (base + j * 32 + lane < n) {
        const int at = mine[(int)((key[j] >> shift) & 255)] + rank[j];
        skeys[at] = key[j];
        svals[at] = val[j];
      }
    }
    __syncthreads();
#pragma unroll
    for (int j = 0; j < kSmallItems; ++j) {
      const int p = base + j * 32 + lane;
      if (p < n) {
        key[j] = skeys[p];
        val[j] = svals[p];
      }
    }
  }
#pragma unroll
  for (int j = 0; j < kSmallItems; ++j) {
    const int p = base + j * 32 + lane;
    if (p < n) {
      if (keys_out != nullptr) keys_out[p] = key[j];
      vals_out[p] = val[j];
    }
  }
}

// Exclusive scan of in[0 .. n) into out, and the sum at out[n].  out is not in (a
// tile whose wait ran out reads what lies before it again).  Sums up to 2^31 - 1 (a
// context holds that many reverse pairs of the nested grids).
constexpr int kScanItems = 16;
constexpr int kScanTile = kScanThreads * kScanItems;

template <class T>
__global__ void __launch_bounds__(kScanThreads)
k_scan(const T* __restrict__ in, int32_t* __restrict__ out, int64_t n, int32_t* __restrict__ ticket, uint64_t* pub) {
  constexpr int kLoad = 16 / (int)sizeof(T);  // items of 16 bytes
  __shared__ int32_t s_tile, s_before;
  const int64_t tiles = n > 0 ? (n + kScanTile - 1) / kScanTile : 1;
  const bool vec = (((uintptr_t)in | (uintptr_t)out) & 15u) == 0u;
  for (;;) {
    if (threadIdx.x == 0) s_tile = atomicAdd(ticket, 1);
    __syncthreads();
    const int32_t tile = s_tile;
    if (tile >= tiles) return;
    const int64_t c0 = (int64_t)tile * kScanTile + threadIdx.x * kScanItems;
    int32_t v[kScanItems];
    if (vec && c0 + kScanItems <= n) {
#pragma unroll
      for (int i = 0; i < kScanItems; i += kLoad) {
        const uint4 q = *reinterpret_cast<const uint4*>(in + c0 + i);
        const uint32_t word[4] = {q.x, q.y, q.z, q.w};
#pragma unroll
        for (int k = 0; k < kLoad; ++k)
          v[i + k] = sizeof(T) == 4 ? (int32_t)word[k & 3] : (int32_t)((word[k >> 2] >> (8 * (k & 3))) & 255u);
      }
    } else {
#pragma unroll
      for (int i = 0; i < kScanItems; ++i) v[i] = c0 + i < n ? (int32_t)in[c0 + i] : 0;
    }
    int32_t s = 0;
#pragma unroll
    for (int i = 0; i < kScanItems; ++i) s += v[i];
    int32_t tot;
    int32_t run = block_scan(s, &tot);
    const int32_t before = tiles_before(pub, tile, tot, (int64_t)tile * kScanTile, &s_before,
                                        [&](int64_t i) { return (int32_t)in[i]; });
    run += before;
    if (tile == tiles - 1 && threadIdx.x == 0) out[n] = before + tot;
    if (vec && c0 + kScanItems <= n) {
#pragma unroll
      for (int i = 0; i < kScanItems; i += 4) {
        int4 q;
        q.x = run;
        q.y = q.x + v[i];
        q.z = q.y + v[i + 1];
        q.w = q.z + v[i + 2];
        run = q.w + v[i + 3];
        *reinterpret_cast<int4*>(out + c0 + i) = q;
      }
    } else {
#pragma unroll
      for (int i = 0; i < kScanItems; ++i) {
        if (c0 + i < n) out[c0 + i] = run;
        run += v[i];
      }
    }
    __syncthreads();  // s_before and s_tile are read before the next tile's
  }
}

}  // namespace sphk

namespace sphh {
using namespace sphk;

// Sort scratch: per pass 256 digit counts, a tile counter and 256 published
// words per tile.
int64_t radix_words(int64_t n, int passes) {
  return (int64_t)passes * (256 + 1 + 256 * ((n + kRadixTile - 1) / kRadixTile)) + 64;
}

template <class K>
static cudaError_t radix_sort_impl(int64_t n, int bits, const K* keys, K* keys_out, K* keys_tmp, bool want_keys,
                                   int32_t* vals_out, int32_t* vals_tmp, int32_t* scratch, cudaStream_t st) {
  if (n <= 0) return cudaSuccess;
  const int64_t tiles = (n + kRadixTile - 1) / kRadixTile;
  const int passes = bits <= 0 ? 1 : (bits + 7) / 8;
  if (passes > kRadixMaxPasses) return cudaErrorInvalidValue;
  if (n <= kSmallMax) {
    static PerDevice<1> known;
    int bytes[1];
    const cudaError_t e = known.get(bytes, [](int (&v)[1]) {
      v[0] = (int)small_smem<K>();
      return opt_in(k_radix_small<K>, small_smem<K>());
    });
    if (e != cudaSuccess) return e;
    const int warps = (int)((n + 32 * kSmallItems - 1) / (32 * kSmallItems));
    k_radix_small<K><<<1, 32 * (warps < 8 ? 8 : warps), small_smem<K>(), st>>>((int)n, keys, passes,
                                                                               want_keys ? keys_out : nullptr, vals_out);
    return cudaGetLastError();
  }
  cudaError_t e = cudaMemsetAsync(scratch, 0, sizeof(int32_t) * (size_t)radix_words(n, passes), st);
  if (e != cudaSuccess) return e;
  int32_t* hist = scratch;
  int32_t* ticket = hist + 256 * passes;
  uint32_t* pub = reinterpret_cast<uint32_t*>(ticket + passes);
  k_radix_hist<K><<<(unsigned)(tiles < 1024 ? tiles : 1024), kScanThreads, 0, st>>>(n, keys, passes, hist);
  const K* k_in = keys;
  const int32_t* v_in = nullptr;
  for (int p = 0; p < passes; ++p) {
    // outputs alternate so that the last pass lands in keys_out / vals_out
    const bool odd = ((passes - 1 - p) & 1) != 0;
    K* k_out = odd ? keys_tmp : keys_out;
    int32_t* v_out = odd ? vals_tmp : vals_out;
    k_radix_pass<K><<<(unsigned)tiles, kScanThreads, 0, st>>>(n, k_in, v_in, 8 * p, hist + 256 * p, ticket + p,
                                                               pub + (int64_t)p * tiles * 256,
                                                               p == passes - 1 && !want_keys ? nullptr : k_out, v_out);
    k_in = k_out;
    v_in = v_out;
  }
  return cudaGetLastError();
}

cudaError_t radix_sort_index(int64_t n, int bits, const int32_t* keys, int32_t* keys_out, int32_t* keys_tmp,
                             int32_t* vals_out, int32_t* vals_tmp, int32_t* scratch, cudaStream_t st) {
  return radix_sort_impl<int32_t>(n, bits, keys, keys_out, keys_tmp, true, vals_out, vals_tmp, scratch, st);
}

cudaError_t radix_sort_index64(int64_t n, int bits, const uint64_t* keys, uint64_t* keys_out, uint64_t* keys_tmp,
                               int32_t* vals_out, int32_t* vals_tmp, int32_t* scratch, cudaStream_t st) {
  return radix_sort_impl<uint64_t>(n, bits, keys, keys_out, keys_tmp, true, vals_out, vals_tmp, scratch, st);
}

cudaError_t radix_partition(int64_t n, const int8_t* keys, int32_t* vals_out, int32_t* scratch, cudaStream_t st) {
  return radix_sort_impl<int8_t>(n, 8, keys, nullptr, nullptr, false, vals_out, nullptr, scratch, st);
}

// the tile counter, and from an 8-byte boundary a published word of 64 bits per tile
int64_t scan_words(int64_t n) { return 2 * ((n + kScanTile - 1) / kScanTile) + 4; }

template <class T>
static cudaError_t scan_impl(const T* in, int32_t* out, int64_t n, int32_t* scratch, int num_sms, cudaStream_t st) {
  const int64_t tiles = n > 0 ? (n + kScanTile - 1) / kScanTile : 1;
  const cudaError_t e = cudaMemsetAsync(scratch, 0, sizeof(int32_t) * (size_t)(2 * tiles + 2), st);
  if (e != cudaSuccess) return e;
  const int64_t most = (int64_t)num_sms * 6;
  k_scan<T><<<(unsigned)(tiles < most ? tiles : most), kScanThreads, 0, st>>>(
      in, out, n, scratch, reinterpret_cast<uint64_t*>(scratch + 2));
  return cudaGetLastError();
}

cudaError_t scan_exclusive(const int32_t* in, int32_t* out, int64_t n, int32_t* scratch, int num_sms,
                           cudaStream_t st) {
  return scan_impl(in, out, n, scratch, num_sms, st);
}

cudaError_t scan_exclusive(const uint8_t* in, int32_t* out, int64_t n, int32_t* scratch, int num_sms,
                           cudaStream_t st) {
  return scan_impl(in, out, n, scratch, num_sms, st);
}

}  // namespace sphh
