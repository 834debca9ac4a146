// tree.cu -- nested grids for inputs whose smoothing lengths span orders of
// magnitude (Sec. 2.1 and Sec. 9.1: a top-level grid whose cells are
// recursively split into 8 children, particles stored depth-first so that
// every cell at every level is a contiguous range, and interactions taken
// between cells of the size that matches the local h).
//
// The top level is the uniform grid of cells.cu (cells >= the largest
// support).  Below each top cell the particles are ordered by the Morton code
// of their position at depth kTreeDepth (1024 sub-cells per side), giving a
// 64-bit source key (top cell id << 30 | Morton code) that the stable radix
// sort orders: "source order".  A cell at depth d is the set of keys sharing
// their top 30 - 3 (kTreeDepth - d) Morton bits, i.e. one contiguous range.
//
// Levels.  A cell holding at most n_leaf particles is not split.  Each
// particle works at its own level: the deepest depth d whose cell side is at
// least (1 + margin) H_i, stopping at a cell with at most n_leaf particles or
// at kTreeDepth.  (A rule on the largest H of a whole cell would keep a dense
// core at the coarse level of the one wide particle beside it; per particle,
// each target's 27 neighbour cells stay ~H wide.)  "Target order" is a stable
// partition of source order by level: the particles of one cell at one level,
// a group, follow each other in it.  (One digit of sorting instead of a second
// 64-bit sort by cell and level, 40 us instead of 390 us at 2M particles; and
// the groups of the coarse levels, whose cells may hold thousands of sources,
// come first, so that the loops do not end on them.)  A group's sources are the particles of the 27 cells of
// its level around it, one source-order range each (binary search), which
// hold every particle within one cell side of the group: enough for the
// density of its targets, whose supports are at most that side.
#include "lookback.cuh"
#include "sph_internal.cuh"
#include "sph_launch.h"
#include "tree.cuh"

namespace sphk {

__global__ void k_tree_key(int64_t n, const double* __restrict__ x, const double* __restrict__ y,
                           const double* __restrict__ z, const int64_t* __restrict__ sim_offset,
                           int n_sims, const GridDev* __restrict__ grid,
                           const int32_t* __restrict__ cell_key, uint64_t* __restrict__ key64) {
  const WarpRange wr = warp_range(n);
  SimCursor sc;
  for (int64_t p = wr.lo + (threadIdx.x & 31); p < wr.hi; p += 32) {
    const int s = sc.at(sim_offset, n_sims, p);
    const GridDev G = grid[s];
    const int32_t c = cell_key[p];
    const int32_t local = c - G.cell_base;
    const int32_t kx = local % G.n_c, ky = (local / G.n_c) % G.n_c, kz = local / (G.n_c * G.n_c);
    const uint32_t lx = (uint32_t)(fine_coord_fast(x[p], G, kx) - kx * kTreeFine);
    const uint32_t ly = (uint32_t)(fine_coord_fast(y[p], G, ky) - ky * kTreeFine);
    const uint32_t lz = (uint32_t)(fine_coord_fast(z[p], G, kz) - kz * kTreeFine);
    const uint64_t k = ((uint64_t)(uint32_t)c << 30) | (spread3(lx) | (spread3(ly) << 1) | (spread3(lz) << 2));
    key64[p] = k;
  }
}

// Level and cell side of each particle (source order), by descending from its
// top cell.
__global__ void k_tree_level(int64_t n, const uint64_t* __restrict__ skey, const int32_t* __restrict__ perm,
                             const float* __restrict__ h, int n_sims,
                             const GridDev* __restrict__ grid, int n_leaf, double margin, float gamma_k,
                             int8_t* __restrict__ level, float* __restrict__ leaf_side) {
  for (int64_t s = (int64_t)blockIdx.x * blockDim.x + threadIdx.x; s < n; s += (int64_t)gridDim.x * blockDim.x) {
    const uint64_t key = skey[s];
    const int32_t c = (int32_t)(key >> 30);
    const GridDev G = grid[sim_of_cell(grid, n_sims, c)];
    const double reach = (1.0 + margin) * (double)(gamma_k * h[perm[s]]);
    // A cell holding s has at most n_leaf particles only if it lies within
    // (s - n_leaf, s + n_leaf) in source order: if the key n_leaf places away
    // on either side shares its prefix, the cell holds more; else its bounds
    // are searched in that window (a few loads near s, instead of bisecting
    // each level's cell from its parent's range)
    const int64_t wl = s - n_leaf, wr = s + n_leaf;
    const uint64_t kl = wl >= 0 ? skey[wl] : 0ull, kr = wr < n ? skey[wr] : 0ull;
    int d = 0;
    // the side of level d + 1, G.cell / 2^(d + 1), by exact halvings (no
    // FP64 division: this GPU's FP64 pipe is slow)
    double side_next = 0.5 * G.cell;
    for (;; ++d, side_next *= 0.5) {
      const int sh = 3 * (kTreeDepth - d);
      const uint64_t pre = key >> sh;
      bool small = false;  // the cell holds at most n_leaf particles
      if (!((wl >= 0 && (kl >> sh) == pre) || (wr < n && (kr >> sh) == pre))) {
        const int64_t lo = lower_bound64(skey, wl + 1 > 0 ? wl + 1 : 0, s + 1, pre << sh);
        const int64_t hi = lower_bound64(skey, s + 1, wr < n ? wr : n, (pre + 1) << sh);
        small = hi - lo <= n_leaf;
      }
      if (d == kTreeDepth || small) break;
      if (side_next < reach) break;
    }
    level[s] = (int8_t)d;
    leaf_side[s] = G.cell_f * __int_as_float((127 - d) << 23);  // G.cell_f / 2^d, exact
  }
}

// The groups in target order: a target whose level or cell differs from the
// one before it starts a group.  Each target's group (leaf_of), the group
// records with a sentinel, and their number; tiles of 2048 targets, prefixed by
// look-back.
constexpr int kLeafItems = 8;
constexpr int kLeafTile = kScanThreads * kLeafItems;
__global__ void __launch_bounds__(kScanThreads)
k_tree_leaves(int64_t n, const int32_t* __restrict__ tgt, const int8_t* __restrict__ level,
              const uint64_t* __restrict__ skey, int32_t* __restrict__ leaf_of, TreeLeaf* __restrict__ leaves,
              int32_t* __restrict__ n_leaves, int32_t* __restrict__ ticket, uint64_t* pub) {
  __shared__ int32_t s_tile, s_before;
  if (threadIdx.x == 0) s_tile = atomicAdd(ticket, 1);
  __syncthreads();
  const int32_t tile = s_tile;
  const int64_t k0 = (int64_t)tile * kLeafTile + threadIdx.x * kLeafItems;
  uint64_t key[kLeafItems];
  int d[kLeafItems];
  unsigned first = 0u;  // bit i: target k0 + i starts a group
  uint64_t cell = 0;
  int last = -1;
  if (k0 > 0 && k0 < n) {
    const int32_t s = tgt[k0 - 1];
    last = level[s];
    cell = skey[s] >> (3 * (kTreeDepth - last));
  }
#pragma unroll
  for (int i = 0; i < kLeafItems; ++i) {
    const int64_t k = k0 + i;
    key[i] = 0;
    d[i] = 0;
    if (k < n) {
      const int32_t s = tgt[k];
      d[i] = level[s];
      key[i] = skey[s];
      const uint64_t c = key[i] >> (3 * (kTreeDepth - d[i]));
      if (d[i] != last || c != cell) first |= 1u << i;
      last = d[i];
      cell = c;
    }
  }
  int32_t tot;
  int32_t at = block_scan(__popc(first), &tot);
  const int32_t before = tiles_before(pub, tile, tot, (int64_t)tile * kLeafTile, &s_before, [&](int64_t k) {
    if (k == 0) return 1;
    const int32_t s = tgt[k], r = tgt[k - 1];
    const int sh = 3 * (kTreeDepth - level[s]);
    return level[s] != level[r] || (skey[s] >> sh) != (skey[r] >> sh) ? 1 : 0;
  });
  at += before;
#pragma unroll
  for (int i = 0; i < kLeafItems; ++i) {
    const int64_t k = k0 + i;
    if (k < n) {
      if ((first >> i) & 1u) {
        TreeLeaf L = cell_at_depth(key[i], d[i]);
        L.start = (int32_t)k;
        leaves[at++] = L;
      }
      leaf_of[k] = at - 1;
    }
  }
  if (threadIdx.x == 0 && ((int64_t)tile + 1) * kLeafTile >= n) {
    const int32_t nl = before + tot;
    *n_leaves = nl;
    leaves[nl].start = (int32_t)n;  // sentinel: end of the last group
  }
}

// 27 neighbour ranges of each leaf: the cells of the leaf's side around it,
// with the periodic shift (-1, 0, +1 boxes) of each axis packed in `shift`.
__global__ void k_tree_neigh(const TreeLeaf* __restrict__ leaves, const int32_t* __restrict__ n_leaves_p,
                             const uint64_t* __restrict__ skey, int64_t n, const int32_t* __restrict__ cell_start,
                             int n_sims, const GridDev* __restrict__ grid, TreeRange* __restrict__ ranges) {
  const int32_t nl = *n_leaves_p;
  for (int64_t t = (int64_t)blockIdx.x * blockDim.x + threadIdx.x; t < (int64_t)nl * 27;
       t += (int64_t)gridDim.x * blockDim.x) {
    const int32_t li = (int32_t)(t / 27);
    const TreeLeaf L = leaves[li];
    const GridDev G = grid[sim_of_cell(grid, n_sims, L.cell)];
    ranges[t] = neighbour_range(G, L, (int)(t % 27), skey, cell_start);
  }
}

// Per particle in tree order: the fine integer position (kTreeFine sub-cells
// per top cell, over the whole box) with the reverse-pair threshold, the FP32 offset from that sub-cell's
// corner (differences of positions stay exact at the leaf scale) with the
// mass, the velocity with u, the starting h, and the list radius
// min(leaf side, kListReach * gamma_K * h).
__global__ void k_tree_gather(int64_t n, const int32_t* __restrict__ perm, const uint64_t* __restrict__ skey,
                              int n_sims, const GridDev* __restrict__ grid, const double* __restrict__ x,
                              const double* __restrict__ y, const double* __restrict__ z,
                              const float* __restrict__ m, const float* __restrict__ vx,
                              const float* __restrict__ vy, const float* __restrict__ vz,
                              const float* __restrict__ u, const float* __restrict__ h,
                              const float* __restrict__ leaf_side, float list_reach, float gamma_k,
                              int4* __restrict__ fine,
                              float4* __restrict__ rel, float4* __restrict__ vel4, float* __restrict__ hs,
                              float* __restrict__ lrad) {
  for (int64_t s = (int64_t)blockIdx.x * blockDim.x + threadIdx.x; s < n; s += (int64_t)gridDim.x * blockDim.x) {
    const int32_t p = perm[s];
    const uint64_t key = skey[s];
    const int32_t c = (int32_t)(key >> 30);
    const GridDev G = grid[sim_of_cell(grid, n_sims, c)];
    const int32_t local = c - G.cell_base, nc = G.n_c;
    const int32_t kx = local % nc, ky = (local / nc) % nc, kz = local / (nc * nc);
    const uint32_t mc = (uint32_t)(key & 0x3fffffffu);
    const int32_t gx = kx * kTreeFine + (int32_t)compact3(mc);
    const int32_t gy = ky * kTreeFine + (int32_t)compact3(mc >> 1);
    const int32_t gz = kz * kTreeFine + (int32_t)compact3(mc >> 2);
    const double sf = G.cell / (double)kTreeFine;
    const float hp = h[p];
    const float R = fminf(leaf_side[s], list_reach * gamma_k * hp);
    // w: the list radius lowered by a margin of the leaf side (the reverse
    // pairs' threshold, read with the fine position)
    fine[s] = make_int4(gx, gy, gz, __float_as_int(R - 0x1p-18f * leaf_side[s]));
    rel[s] = make_float4((float)(x[p] - (double)gx * sf), (float)(y[p] - (double)gy * sf),
                         (float)(z[p] - (double)gz * sf), m[p]);
    vel4[s] = make_float4(vx[p], vy[p], vz[p], u[p]);
    hs[s] = hp;
    lrad[s] = R;
  }
}

}  // namespace sphk

namespace sphh {
using namespace sphk;

static int blocks_n(int64_t n) {
  int64_t b = (n + 255) / 256;
  return (int)(b < 1 ? 1 : (b > 65535 ? 65535 : b));
}

cudaError_t launch_tree_build(const TreeBuildArgs& a, cudaStream_t st) {
  const int64_t n = a.n_total;
  cudaError_t e;
  if (n <= 0) {
    e = cudaMemsetAsync(a.n_leaves, 0, sizeof(int32_t), st);
    return e != cudaSuccess ? e : launch_cell_bounds(0, a.skey, 30, a.cap_cells, a.num_sms, a.misc, a.cell_start, st);
  }
  int cbits = 1;
  while (cbits < 30 && ((int64_t)1 << cbits) <= a.cap_cells) ++cbits;
  // source order: (top cell, Morton code), ties by pool index
  k_tree_key<<<blocks_n(n), 256, 0, st>>>(n, a.x, a.y, a.z, a.sim_offset, a.n_sims, a.grid, a.cell_key, a.key64);
  e = radix_sort_index64(n, 30 + cbits, a.key64, a.skey, a.key64_b, a.perm, a.rv, a.hist, st);
  if (e != cudaSuccess) return e;
  e = launch_cell_bounds(n, a.skey, 30, a.cap_cells, a.num_sms, a.misc, a.cell_start, st);
  if (e != cudaSuccess) return e;
  // levels, and target order: by level, ties by source index
  k_tree_level<<<blocks_n(n), 256, 0, st>>>(n, a.skey, a.perm, a.h, a.n_sims, a.grid, a.n_leaf, a.margin, a.gamma_k,
                                            a.level, a.leaf_side);
  e = radix_partition(n, a.level, a.tgt, a.hist, st);
  if (e != cudaSuccess) return e;
  const int64_t tiles = (n + kLeafTile - 1) / kLeafTile;
  e = cudaMemsetAsync(a.scan_tmp, 0, sizeof(int32_t) * (size_t)(2 * tiles + 2), st);
  if (e != cudaSuccess) return e;
  k_tree_leaves<<<(unsigned)tiles, kScanThreads, 0, st>>>(n, a.tgt, a.level, a.skey, a.leaf_of, a.leaves, a.n_leaves,
                                                         a.scan_tmp, reinterpret_cast<uint64_t*>(a.scan_tmp + 2));
  k_tree_neigh<<<blocks_n(n * 4), 256, 0, st>>>(a.leaves, a.n_leaves, a.skey, n, a.cell_start, a.n_sims, a.grid,
                                                a.ranges);
  return cudaGetLastError();
}

cudaError_t launch_tree_gather(const TreeGatherArgs& a, cudaStream_t st) {
  if (a.n_total <= 0) return cudaSuccess;
  k_tree_gather<<<blocks_n(a.n_total), 256, 0, st>>>(a.n_total, a.perm, a.skey, a.n_sims, a.grid, a.x, a.y, a.z,
                                                     a.m, a.vx, a.vy, a.vz, a.u, a.h, a.leaf_side, a.list_reach,
                                                     a.gamma_k, a.fine, a.rel, a.vel4, a.hs, a.lrad);
  return cudaGetLastError();
}

}  // namespace sphh
