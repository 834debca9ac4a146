// stencil.cuh -- the 27-cell neighbourhood of a target cell on the uniform
// periodic grid (Sec. 2.1: every neighbour of a particle lies in its own cell
// or one of the 26 adjacent cells, because cells are at least H wide), and the
// warp-cooperative staging of those cells' particles into shared memory.
#pragma once
#include "sph_internal.cuh"

namespace sphk {

// Lane k < 27 of a warp describes neighbour k = (dx+1) + 3 (dy+1) + 9 (dz+1):
// its sorted range and the offset of its particles' cell-relative positions
// when seen from the target cell (a periodic image is just another offset).
struct NbLane {
  int32_t start, len;
  float ox, oy, oz;
};

__device__ __forceinline__ NbLane neighbour_lane(int lane, int32_t cell_base, int32_t cx, int32_t cy,
                                                 int32_t cz, int32_t nc, float cell,
                                                 const int32_t* __restrict__ cell_start) {
  NbLane r;
  r.start = 0;
  r.len = 0;
  r.ox = r.oy = r.oz = 0.0f;
  if (lane < 27) {
    const int dx = lane % 3 - 1, dy = (lane / 3) % 3 - 1, dz = lane / 9 - 1;
    int32_t nx = cx + dx, ny = cy + dy, nz = cz + dz;
    nx += nx < 0 ? nc : 0;
    nx -= nx >= nc ? nc : 0;
    ny += ny < 0 ? nc : 0;
    ny -= ny >= nc ? nc : 0;
    nz += nz < 0 ? nc : 0;
    nz -= nz >= nc ? nc : 0;
    const int32_t nbc = cell_base + nx + nc * (ny + nc * nz);
    r.start = cell_start[nbc];
    r.len = cell_start[nbc + 1] - r.start;
    r.ox = (float)dx * cell;
    r.oy = (float)dy * cell;
    r.oz = (float)dz * cell;
  }
  return r;
}

__device__ __forceinline__ int warp_sum_int(int v) {
#pragma unroll
  for (int o = 16; o > 0; o >>= 1) v += __shfl_xor_sync(0xffffffffu, v, o);
  return v;
}

// Copies the virtual source range [v0, v0 + cap) of the concatenation of the
// 27 neighbour cells into shared memory through `put(slot, j, ox, oy, oz)`.
// Returns the number of sources staged.  Warp-collective.
template <class Put>
__device__ __forceinline__ int stage_sources(int v0, int cap, const NbLane& nb, int lane, Put put) {
  int cum = 0;
#pragma unroll 1
  for (int k = 0; k < 27; ++k) {
    const int32_t st = __shfl_sync(0xffffffffu, nb.start, k);
    const int32_t len = __shfl_sync(0xffffffffu, nb.len, k);
    const float ox = __shfl_sync(0xffffffffu, nb.ox, k);
    const float oy = __shfl_sync(0xffffffffu, nb.oy, k);
    const float oz = __shfl_sync(0xffffffffu, nb.oz, k);
    const int lo = max(v0, cum), hi = min(v0 + cap, cum + len);
    for (int v = lo + lane; v < hi; v += 32) put(v - v0, st + (v - cum), ox, oy, oz);
    cum += len;
  }
  __syncwarp();
  return min(cum, v0 + cap) - v0;
}

// ---- cells of blocks that do not fit the loops' staging (overflow kernels) ----
//
// A CTA of kWarpsPerBlock warps per target cell.  The sources of the 27 cells
// (up to 768 for the density, 640 for the force) are staged once for all its
// targets; the warps list for each target the staged sources that can count (the
// density: within the cell side, which caps every support; the force: within the
// pair's reach, whatever the supports are), a ballot per target and 32 sources, so
// in the sources' order, and one lane per target walks its list in that order.  A
// source not listed adds exactly zero to every sum, so the sums are those of a walk
// of every source, bit for bit.  More sources than fit are streamed through a buffer
// per warp, 32 targets at a time.
//
// The walks are serial and bound by latency.  Up to one cell per resident CTA
// ("spread") the targets are dealt to the CTA's warps.  With more cells than
// that, issue slots count: the density's lists are walked by one warp, and the
// force, which has one pass over the sources and no more, goes back to a warp
// per cell that streams.  A warp per cell streaming throughout took, density +
// force, 94 + 71 us in a step of 4096 particles (19 per cell, just past the
// blocks' staging; few cells), this 33 + 29; in a pool of 64 lattice boxes (more
// cells than CTAs) 304 + 151 us, this 190 + 170 (the force lists walked by one
// warp: 208; spread there, too: 262 + 295).
constexpr int kOvfList = 128;   // list entries per target; longer: the target walks every staged source
struct OvfLists {
  uint16_t entry[32][kOvfList];
  int count[32];
};

// Stages all nsrc sources (each warp a part) through put(slot, j,
// ox, oy, oz).  CTA-collective, ends with a barrier.
template <class Put>
__device__ __forceinline__ void stage_all(int nsrc, const NbLane& nb, int warp, int lane, Put put) {
  const int part = (nsrc + kWarpsPerBlock - 1) / kWarpsPerBlock, v0 = warp * part;
  if (v0 < nsrc)
    stage_sources(v0, part, nb, lane, [&](int slot, int32_t j, float ox, float oy, float oz) { put(v0 + slot, j, ox, oy, oz); });
  __syncthreads();
}

// Lists of nt <= 32 targets (pos(t) and the staged src[k]: x, y, z and a value):
// the staged slots with r^2 < reach2(pos(t).w, src[k].w), and their counts.
// CTA-collective, ends with a barrier.
template <class Pos, class Reach2>
__device__ __forceinline__ void list_sources(int nt, int nsrc, const float4* src, OvfLists& lists, int warp, int lane,
                                             Pos pos, Reach2 reach2) {
  const unsigned lt = (1u << lane) - 1u;
#pragma unroll 1
  for (int t = warp; t < nt; t += kWarpsPerBlock) {
    const float4 p = pos(t);
    int cnt = 0;
#pragma unroll 1
    for (int v = 0; v < nsrc; v += 32) {
      const float4 q = src[min(v + lane, nsrc - 1)];
      const float dx = p.x - q.x, dy = p.y - q.y, dz = p.z - q.z;
      const bool in = v + lane < nsrc && fmaf(dx, dx, fmaf(dy, dy, dz * dz)) < reach2(p.w, q.w);
      const unsigned m = __ballot_sync(0xffffffffu, in);
      const int at = cnt + __popc(m & lt);
      if (in && at < kOvfList) lists.entry[t][at] = (uint16_t)(v + lane);
      cnt += __popc(m);
    }
    if (lane == 0) lists.count[t] = cnt;
  }
  __syncthreads();
}

// The target of a lane's walk, or -1.
__device__ __forceinline__ int walk_target(bool spread, int nt, int warp, int lane) {
  const int t = spread ? lane * kWarpsPerBlock + warp : (warp == 0 ? lane : 32);
  return t < nt ? t : -1;
}

}  // namespace sphk
