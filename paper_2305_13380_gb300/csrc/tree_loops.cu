// tree_loops.cu -- density and force loops on the leaves of the nested grids
// (tree.cu).  Same mathematics as density.cu / force.cu (Sec. 3.1 and 3.2);
// the unit of work is a leaf and the 27 cells of its size around it.
//
// Positions.  Every particle carries its fine integer position (1024
// sub-cells per top cell) and its FP32 offset from that sub-cell's corner.
// Relative to a leaf corner a position is
//     (fine - corner + shift * N_fine) * s_fine + offset,
// the integer part exact, so FP32 keeps the sub-cell scale's precision
// however wide the top cells are.
//
// Density, a warp per round of kTPer targets of one leaf, kTreeTpp lanes per
// target (k_tree_density):
//   1. filter: the children of the 27 cells that some target of the round
//      reaches, as segments of source order, 32 sources at a time, one per
//      lane, each tested against the round's targets in turn.  The sources
//      closer than a target's list radius R_i = min(leaf side, kTreeListReach *
//      starting support) are kept in shared memory and listed per lane;
//   2. Newton-Raphson passes walk the lists; a target whose support outgrows
//      R_i (or whose list overflows) leaves its round for the per-target kernel
//      (k_tree_density_fb at its own level: a warp per target over its 27
//      cells), so that its round-mates do not wait;
//   3. the final pass at the converged h gathers the sources from memory and
//      publishes the lists for the force loop.
// A force pair needs r < max(H_i, H_j).  The list of i holds every j with
// r < R_i >= H_i; a j with H_j > r >= R_i is only in j's own reach, so the
// density of j emits it as a reverse pair (receiver i, source j).  Reverse
// pairs are grouped by receiver and sorted by source (deterministic order).
//
// Force, a warp per four targets: each walks its list and its reverse pairs.
// The same kernels run the SPHENIX force and gradient pass (Sec. 3.3) with a
// fifth record per source (kTSphenix, kTGradient).
// Whether a pair is the list's or a reverse pair is decided in the target's
// own leaf frame with the same arithmetic as the density filter, so no pair is
// counted twice or dropped at the boundary; emission uses a margin so that the
// reverse pairs are a superset.
#include "per_device.h"
#include "sph_internal.cuh"
#include "sph_launch.h"
#include "tree.cuh"

namespace sphk {

constexpr int kTWarps = 4;             // warps per CTA
constexpr int kTCap = 320;             // staged sources per warp and chunk (per-target kernel)
constexpr int kTPer = 32 / kTreeTpp;   // targets per round
constexpr int kTChildren = 27 * 8;     // children of the 27 neighbour cells

// Tables of a warp's leaf.
struct TTab {
  int32_t cv[kTChildren + 1];          // virtual start of each child (Morton order), + end
  int32_t rlo[28], rcum[28], rsc[28];  // per neighbour range: first source, virtual start, shift
  uint32_t cact[(kTChildren + 31) / 32];  // masked loops: children holding a masked source
};
// ... and of the per-target kernel.
struct TPrune : TTab {
  int32_t hoff[kTChildren + 4];  // offsets of the target's hit children, + total
  uint8_t hch[kTChildren];       // the hit children, in order
  // ... and their sources: item u's index is x + u, its position relative to the
  // target's cell its fine integer position plus (y, z, w)
  alignas(16) int4 src[kTChildren];
};
constexpr size_t kTPruneBytes = (sizeof(TPrune) + 15) / 16 * 16;
constexpr size_t kTFbWarpSmem = (size_t)kTCap * (sizeof(float4) + sizeof(uint32_t)) + kTPruneBytes;
constexpr size_t kTFbSmem = kTWarps * kTFbWarpSmem;
static_assert(kTFbWarpSmem % 16 == 0, "per-warp regions keep float4 alignment");

// A density warp's shared memory.  Only the sources that some target of the
// round lists are kept (about 90 of the ~305 it tests), as a position and a
// packed index, and a list entry is one byte, the slot.
constexpr int kTKept = 256;
constexpr int kTWhole = 384;           // a leaf with at most this many sources is taken whole
constexpr int kTSegs = 27 * 4 + 4;     // runs of hit children: at most four per range
constexpr int kTWin = 2 * kTPer;       // targets per window (k_tree_density)
// resident CTAs per SM that the registers are sized for (the plain instance over
// 2M clustered particles: 5 4.18, 6 3.85, 7 3.88 ms; the masked one, which keeps
// more alive, over 1M: 4 734, 5 657, 6 734 us)
constexpr int kTDensBlocks = 6, kTMaskBlocks = 5;
struct TRound {
  float4 pos[kTKept];                  // position from the leaf corner; packed index and shift
  float4 tgt[kTPer];                   // the targets' positions and R^2
  int2 seg[kTSegs];                    // segments: virtual start; first source and shift
  TTab tab;
  uint8_t list[kTreeList + 1][32];     // + one scratch row for an overflowing append
};
constexpr size_t kTRoundBytes = (sizeof(TRound) + 15) / 16 * 16;
constexpr size_t kTDensSmem = kTWarps * kTRoundBytes;
static_assert(kTDensBlocks * (kTDensSmem + 1024) <= 228 * 1024, "resident density CTAs per SM");
static_assert(kTKept <= 256 && kTreeTpp * kTreeList <= kTKept, "a slot is a byte; one target's list fits");
// the sources of lane sub among 32: bits sub, sub + kTreeTpp, ...
constexpr uint32_t kTLanes = 0x01010101u;
constexpr uint32_t kTGroup = (1u << kTreeTpp) - 1u;  // the lanes of one target
static_assert(kTreeTpp == 8 && kTreeList == 32, "one byte per target in a ballot, one mark bit per entry");
constexpr int kNoShift = 1 | (1 << 2) | (1 << 4);
// list_cnt marker: the target is solved by the per-target kernels
constexpr uint16_t kListFallback = 0xfffe;
// fallback queue entries: a target index, with this bit for a target queued
// from its group (solved at its own level), and this one for a target outside
// the mask of masked loops (its current support sends reverse pairs only);
// indices stay below 2^29
constexpr int32_t kFbOwnLevel = 1 << 30;
constexpr int32_t kFbPassive = 1 << 29;
constexpr int32_t kFbIndex = kFbPassive - 1;
static_assert(kTreeList <= kTreeListRegion, "published lists fit their regions");
// a target's published list: its lanes' first entries, then their second ones,
// and so on, in a region of kTreeTpp * kTreeListRegion entries, the count in list_cnt[target]
constexpr int kTreeListTarget = kTreeTpp * kTreeListRegion;

struct TGeo {
  float s_fine;        // side of a fine sub-cell
  float side;          // side of the leaf
  double side_d;
  int32_t nfine;       // fine sub-cells per box side
  int32_t ox, oy, oz;  // fine integer position of the leaf corner
  double L;
};

__device__ __forceinline__ TGeo leaf_geo(const TreeLeaf& Lf, const GridDev& G) {
  TGeo g;
  const int32_t local = Lf.cell - G.cell_base, nc = G.n_c;
  const int32_t kx = local % nc, ky = (local / nc) % nc, kz = local / (nc * nc);
  const int sh = kTreeDepth - Lf.depth;
  g.ox = kx * kTreeFine + (Lf.lx << sh);
  g.oy = ky * kTreeFine + (Lf.ly << sh);
  g.oz = kz * kTreeFine + (Lf.lz << sh);
  g.s_fine = (float)(G.cell / (double)kTreeFine);
  g.side_d = G.cell * __longlong_as_double((long long)(1023 - Lf.depth) << 52);  // G.cell / 2^depth, exact
  g.side = (float)g.side_d;
  g.nfine = nc * kTreeFine;
  g.L = G.L;
  return g;
}

// Position relative to the leaf corner of a particle seen with periodic shift
// code sc (2 bits per axis, shift + 1).
__device__ __forceinline__ float3 rel_to(const TGeo& g, const float4& rel, const int4& fine, int sc) {
  const int sx = (sc & 3) - 1, sy = ((sc >> 2) & 3) - 1, sz = ((sc >> 4) & 3) - 1;
  const int32_t dx = fine.x - g.ox + sx * g.nfine;
  const int32_t dy = fine.y - g.oy + sy * g.nfine;
  const int32_t dz = fine.z - g.oz + sz * g.nfine;
  return make_float3(fmaf((float)dx, g.s_fine, rel.x), fmaf((float)dy, g.s_fine, rel.y),
                     fmaf((float)dz, g.s_fine, rel.z));
}

__device__ __forceinline__ float r2_of(const float3& a, const float4& b) {
  const float dx = a.x - b.x, dy = a.y - b.y, dz = a.z - b.z;
  return fmaf(dx, dx, fmaf(dy, dy, dz * dz));
}

// Pair vector x_i - x_j with the exact integer part (sc = shift code of j).
__device__ __forceinline__ float3 pair_vec(const TGeo& g, const float4& rel_i, const int4& fine_i,
                                           const float4& rel_j, const int4& fine_j, int sc) {
  const int sx = (sc & 3) - 1, sy = ((sc >> 2) & 3) - 1, sz = ((sc >> 4) & 3) - 1;
  const int32_t dx = fine_i.x - fine_j.x - sx * g.nfine;
  const int32_t dy = fine_i.y - fine_j.y - sy * g.nfine;
  const int32_t dz = fine_i.z - fine_j.z - sz * g.nfine;
  return make_float3(fmaf((float)dx, g.s_fine, rel_i.x - rel_j.x), fmaf((float)dy, g.s_fine, rel_i.y - rel_j.y),
                     fmaf((float)dz, g.s_fine, rel_i.z - rel_j.z));
}

// List entries pack the tree-order index (26 bits) with the shift code.
__device__ __forceinline__ uint32_t pack_js(int32_t j, int sc) { return (uint32_t)j | ((uint32_t)sc << 26); }
__device__ __forceinline__ int32_t unpack_j(uint32_t e) { return (int32_t)(e & 0x3ffffffu); }
__device__ __forceinline__ int unpack_s(uint32_t e) { return (int)(e >> 26); }
// Shift code of i seen from j, given that of j seen from i.
__device__ __forceinline__ int mirror_s(int sc) {
  return (2 - (sc & 3)) | ((2 - ((sc >> 2) & 3)) << 2) | ((2 - ((sc >> 4) & 3)) << 4);
}

// Groups are handed out one per warp from a counter: their costs differ by
// orders of magnitude (a coarse group beside a dense core stages thousands of
// sources), so a static assignment leaves a few warps running long after the
// others are done.
__device__ __forceinline__ int32_t next_group(int32_t* work, int lane) {
  int32_t g = 0;
  if (lane == 0) g = atomicAdd(work, 1);
  return __shfl_sync(0xffffffffu, g, 0);
}

struct TDSums {
  float w, dw, mw, mdw, div, cx, cy, cz;
  int npair;
};

__device__ __forceinline__ void tds_zero(TDSums& s) {
  s.w = s.dw = s.mw = s.mdw = s.div = s.cx = s.cy = s.cz = 0.f;
  s.npair = 0;
}

// One density pair with x_ij = (dx, dy, dz) (same terms as density.cu).
template <int K>
__device__ __forceinline__ void tdens_pair(float dx, float dy, float dz, const float4& vi, const float4& vj,
                                           float mj, float H, float Hinv, TDSums& s) {
  const float r2 = fmaf(dx, dx, fmaf(dy, dy, dz * dz));
  const float rinv = rsqrt_norm(fmaxf(r2, 1e-30f));
  const float q = r2 * rinv * Hinv;
  float w, g;
  kernel_w_g<K>(q, H * rinv, w, g);
  const float dw = fmaf(q * q, g, 3.0f * w);
  s.w += w;
  s.dw += dw;
  s.mw = fmaf(mj, w, s.mw);
  s.mdw = fmaf(mj, dw, s.mdw);
  const float ux = vj.x - vi.x, uy = vj.y - vi.y, uz = vj.z - vi.z;
  const float mg = mj * g;
  s.div = fmaf(mg, fmaf(ux, dx, fmaf(uy, dy, uz * dz)), s.div);
  s.cx = fmaf(mg, fmaf(uz, dy, -uy * dz), s.cx);
  s.cy = fmaf(mg, fmaf(ux, dz, -uz * dx), s.cy);
  s.cz = fmaf(mg, fmaf(uy, dx, -ux * dy), s.cz);
  s.npair += q < 1.0f;
}

// n-hat and its h-derivative terms of one pair (Newton passes).
template <int K>
__device__ __forceinline__ void tnewton_pair(float r2, float H, float Hinv, float& Sw, float& Sdw) {
  const float rinv = rsqrt_norm(fmaxf(r2, 1e-30f));
  const float q = r2 * rinv * Hinv;
  float w, dw;
  kernel_w_dw<K>(q, w, dw);
  Sw += w;
  Sdw += dw;
}

// Sum over the kTreeTpp lanes of a target (called by all 32 lanes).
__device__ __forceinline__ float gsum(float v) {
#pragma unroll
  for (int o = 1; o < kTreeTpp; o <<= 1) v += __shfl_xor_sync(0xffffffffu, v, o);
  return v;
}

__device__ __forceinline__ int gsumi(int v) {
#pragma unroll
  for (int o = 1; o < kTreeTpp; o <<= 1) v += __shfl_xor_sync(0xffffffffu, v, o);
  return v;
}

__device__ __forceinline__ float gmax(float v) {
#pragma unroll
  for (int o = 1; o < kTreeTpp; o <<= 1) v = fmaxf(v, __shfl_xor_sync(0xffffffffu, v, o));
  return v;
}

// True for every lane of a target if any of its lanes has b (called by all
// 32 lanes).
__device__ __forceinline__ bool group_any(bool b, int lane) {
  const unsigned m = __ballot_sync(0xffffffffu, b);
  return ((m >> (lane & ~(kTreeTpp - 1))) & ((1u << kTreeTpp) - 1u)) != 0u;
}

__device__ __forceinline__ void tcombine(TDSums& s) {
  s.w = gsum(s.w);
  s.dw = gsum(s.dw);
  s.mw = gsum(s.mw);
  s.mdw = gsum(s.mdw);
  s.div = gsum(s.div);
  s.cx = gsum(s.cx);
  s.cy = gsum(s.cy);
  s.cz = gsum(s.cz);
  s.npair = gsumi(s.npair);
}

// The leaf's 27 ranges, lane r < 27 holding range r; lanes 27..31 hold empty
// ranges, so lane 27's cumulative start is the total.
struct TRanges {
  int32_t lo, cum, sc;
  int nsrc;
};

__device__ __forceinline__ TRanges load_ranges(const TreeRange* __restrict__ ranges, int32_t li, int lane) {
  TRanges R;
  int32_t len = 0;
  R.lo = 0;
  R.sc = kNoShift;
  if (lane < 27) {
    const TreeRange t = ranges[(int64_t)li * 27 + lane];
    R.lo = t.lo;
    len = t.hi - t.lo;
    R.sc = t.shift;
  }
  int incl = len;
#pragma unroll
  for (int o = 1; o < 32; o <<= 1) {
    const int v = __shfl_up_sync(0xffffffffu, incl, o);
    if (lane >= o) incl += v;
  }
  R.cum = incl - len;
  R.nsrc = __shfl_sync(0xffffffffu, incl, 31);
  return R;
}

// Pruning tables of a group: per neighbour range its first source, virtual
// start and shift, and the virtual start of each of its 8 children (which
// are contiguous in Morton order; a cell of the deepest level has one).
// Lanes 0..26 search their range's keys.  Called by the whole warp.
__device__ __noinline__ void prune_tables(const uint64_t* __restrict__ skey, TRanges R, int depth,
                                          int lane, TTab* pr, const int32_t* __restrict__ act_pre = nullptr) {
  const int32_t cum_next = __shfl_down_sync(0xffffffffu, R.cum, 1);
  if (act_pre != nullptr) {
    if (lane < (kTChildren + 31) / 32) pr->cact[lane] = 0u;
    __syncwarp();
  }
  if (lane < 27) {
    const int32_t len = cum_next - R.cum;
    pr->rlo[lane] = R.lo;
    pr->rcum[lane] = R.cum;
    pr->rsc[lane] = R.sc;
    int32_t* cvr = pr->cv + lane * 8;
    cvr[0] = R.cum;
    if (depth < kTreeDepth && len > 0) {
      const int sh = 3 * (kTreeDepth - depth - 1);
      const uint64_t base = (skey[R.lo] >> (sh + 3)) << (sh + 3);
      // the seven child boundaries bisected together: each round takes one
      // step of every search, so its loads are in flight at once (a chain of
      // log2(len) loads instead of seven such chains)
      int32_t lo[7], hi[7];
#pragma unroll
      for (int c = 0; c < 7; ++c) {
        lo[c] = R.lo;
        hi[c] = R.lo + len;
      }
#pragma unroll 1
      for (bool more = true; more;) {
        more = false;
#pragma unroll
        for (int c = 0; c < 7; ++c) {
          if (lo[c] < hi[c]) {
            const int32_t mid = (int32_t)(((uint32_t)lo[c] + (uint32_t)hi[c]) >> 1);
            if (skey[mid] < base + ((uint64_t)(c + 1) << sh)) lo[c] = mid + 1; else hi[c] = mid;
            more = more || lo[c] < hi[c];
          }
        }
      }
#pragma unroll
      for (int c = 0; c < 7; ++c) cvr[c + 1] = R.cum + (lo[c] - R.lo);
    } else {
      for (int c = 1; c < 8; ++c) cvr[c] = R.cum + len;
    }
    if (act_pre != nullptr) {
      // which children hold a masked source (prefix sums over the range)
      unsigned bits = 0u;
      int32_t a0 = act_pre[R.lo];
      for (int c = 0; c < 8; ++c) {
        const int32_t v1 = c < 7 ? cvr[c + 1] : R.cum + len;
        const int32_t a1 = act_pre[R.lo + (v1 - R.cum)];
        bits |= (a1 > a0 ? 1u : 0u) << c;
        a0 = a1;
      }
      // 8 children of range `lane` are bits 8 lane .. 8 lane + 7
      if (bits) atomicOr(&pr->cact[lane >> 2], bits << (8 * (lane & 3)));
    }
  }
  if (lane == 0) pr->cv[kTChildren] = R.nsrc;
  __syncwarp();
}

// Squared distance from p (relative to the group corner) to child ch's box:
// neighbour r = ch / 8 at offset (r % 3, r / 3 % 3, r / 9) - 1 cells, child
// bits (x, y, z) = bits 0, 1, 2 of ch % 8, child side cside.
__device__ __forceinline__ float child_dist2(int ch, float side, float cside, const float3& p) {
  const int r = ch >> 3, c = ch & 7;
  const float bx = (float)(r % 3 - 1) * side + (float)(c & 1) * cside;
  const float by = (float)((r / 3) % 3 - 1) * side + (float)((c >> 1) & 1) * cside;
  const float bz = (float)(r / 9 - 1) * side + (float)((c >> 2) & 1) * cside;
  const float ex = fmaxf(fmaxf(bx - p.x, p.x - (bx + cside)), 0.0f);
  const float ey = fmaxf(fmaxf(by - p.y, p.y - (by + cside)), 0.0f);
  const float ez = fmaxf(fmaxf(bz - p.z, p.z - (bz + cside)), 0.0f);
  return fmaf(ex, ex, fmaf(ey, ey, ez * ez));
}

// The children that a target at pi reaches within Rb2 (the per-target kernel):
// lane sub of each eight tests child sub of the 27 cells; the hit children are
// compacted in child order with the offsets of their sources.  Returns their
// number and their sources.  Called by the whole warp.
__device__ __noinline__ int2 prune_round(int lane, float3 pi, float Rb2, const TGeo& g, float cside, TPrune* pr) {
  const float side = g.side;
  uint32_t mine = 0;
  const int sub = lane % kTreeTpp;
#pragma unroll 1
  for (int m = 0; m < 27; ++m) {
    const int ch = 8 * m + sub;
    if (pr->cv[ch] < pr->cv[ch + 1] && child_dist2(ch, side, cside, pi) < Rb2) mine |= 1u << m;
  }
  int nh = 0;
#pragma unroll 1
  for (int m = 0; m < 27; ++m) {
    const bool hb = lane < kTreeTpp && ((mine >> m) & 1u);
    const unsigned b = __ballot_sync(0xffffffffu, hb);
    if (hb) {
      const int ch = 8 * m + lane;
      const int idx = nh + __popc(b & ((1u << lane) - 1u));
      pr->hch[idx] = (uint8_t)ch;
      pr->hoff[idx] = pr->cv[ch + 1] - pr->cv[ch];
    }
    nh += __popc(b);
  }
  __syncwarp();
  int run = 0;
#pragma unroll 1
  for (int k0 = 0; k0 < nh; k0 += 32) {
    const int k = k0 + lane;
    const int v = k < nh ? pr->hoff[k] : 0;
    int incl = v;
#pragma unroll
    for (int o = 1; o < 32; o <<= 1) {
      const int w = __shfl_up_sync(0xffffffffu, incl, o);
      if (lane >= o) incl += w;
    }
    if (k < nh) {
      const int off = run + incl - v, ch = pr->hch[k], r = ch >> 3, sc = pr->rsc[r];
      const int sx = (sc & 3) - 1, sy = ((sc >> 2) & 3) - 1, sz = ((sc >> 4) & 3) - 1;
      pr->hoff[k] = off;
      pr->src[k] = make_int4(pr->rlo[r] + (pr->cv[ch] - pr->rcum[r]) - off, sx * g.nfine - g.ox, sy * g.nfine - g.oy,
                             sz * g.nfine - g.oz);
    }
    run += __shfl_sync(0xffffffffu, incl, 31);
  }
  if (lane == 0) pr->hoff[nh] = run;
  __syncwarp();
  return make_int2(nh, run);
}

// The lane's candidate children of a leaf (child sub of range m: bit m): those
// holding a source, and (mask_only) a masked one (a target outside the mask
// lists only those).  Called once per leaf, after prune_tables.
__device__ __forceinline__ uint32_t group_candidates(int sub, const TTab* pr, bool mask_only) {
  uint32_t c = 0;
#pragma unroll 3
  for (int m = 0; m < 27; ++m) {
    const int ch = 8 * m + sub;
    if (pr->cv[ch] < pr->cv[ch + 1] && (!mask_only || ((pr->cact[ch >> 5] >> (ch & 31)) & 1u))) c |= 1u << m;
  }
  return c;
}

// The segments of a round: the union over its targets of the candidate
// children that they reach, in child order, adjacent children of a range
// (contiguous in source order) as one segment: virtual start and packed first
// source.  The box distances are taken per axis: along each axis a lane's
// child boxes take three positions (the neighbour offset, its child bit
// fixed), so nine squared distances give all 27 (the sum's rounding lies far
// inside the margin of Rb2).  Lane r < 27 then collects the hit children of
// range r from the lanes' masks.  Returns the segments and their sources.  Called
// by the whole warp.
__device__ __noinline__ int2 prune_round_fast(bool valid, int sub, int lane, float3 pi, float Rb2, float side,
                                              float cside, const TTab* pr, uint32_t cand, int2* seg) {
  uint32_t mine = 0;
  if (valid) {
    const float cx = (float)(sub & 1) * cside, cy = (float)((sub >> 1) & 1) * cside, cz = (float)(sub >> 2) * cside;
    float ex[3], ey[3], ez[3];
#pragma unroll
    for (int o = 0; o < 3; ++o) {
      const float b0 = (float)(o - 1) * side;
      const float dx = fmaxf(fmaxf(b0 + cx - pi.x, pi.x - (b0 + cx + cside)), 0.0f);
      const float dy = fmaxf(fmaxf(b0 + cy - pi.y, pi.y - (b0 + cy + cside)), 0.0f);
      const float dz = fmaxf(fmaxf(b0 + cz - pi.z, pi.z - (b0 + cz + cside)), 0.0f);
      ex[o] = dx * dx;
      ey[o] = dy * dy;
      ez[o] = dz * dz;
    }
#pragma unroll
    for (int m = 0; m < 27; ++m)
      if (((cand >> m) & 1u) && ex[m % 3] + ey[(m / 3) % 3] + ez[m / 9] < Rb2) mine |= 1u << m;
  }
#pragma unroll
  for (int o = kTreeTpp; o < 32; o <<= 1) mine |= __shfl_xor_sync(0xffffffffu, mine, o);
  uint32_t hit = 0;
#pragma unroll
  for (int c = 0; c < kTreeTpp; ++c) hit |= ((__shfl_sync(0xffffffffu, mine, c) >> lane) & 1u) << c;
  const int r = lane < 27 ? lane : 0;
  if (lane >= 27) hit = 0;
  const int32_t* cv = pr->cv + 8 * r;
  int len = 0;
#pragma unroll 1
  for (uint32_t b = hit; b != 0u;) {  // the runs of hit children
    const int c0 = __ffs((int)b) - 1, c1 = c0 + __ffs((int)~(b >> c0)) - 1;
    len += cv[c1] - cv[c0];
    b &= b + (1u << c0);
  }
  const int ns = __popc(hit & ~(hit << 1));
  int il = len, in = ns;
#pragma unroll
  for (int o = 1; o < 32; o <<= 1) {
    const int ul = __shfl_up_sync(0xffffffffu, il, o), un = __shfl_up_sync(0xffffffffu, in, o);
    if (lane >= o) {
      il += ul;
      in += un;
    }
  }
  const int2 out = make_int2(__shfl_sync(0xffffffffu, in, 31), __shfl_sync(0xffffffffu, il, 31));
  il -= len;
  in -= ns;
#pragma unroll 1
  for (uint32_t b = hit; b != 0u; ++in) {
    const int c0 = __ffs((int)b) - 1, c1 = c0 + __ffs((int)~(b >> c0)) - 1;
    seg[in] = make_int2(il, (int)pack_js(pr->rlo[r] + (cv[c0] - pr->rcum[r]), pr->rsc[r]));
    il += cv[c1] - cv[c0];
    b &= b + (1u << c0);
  }
  return out;
}

// The hit child (position in the tables) of item u0 + lane of a target's hit
// children; ci: the last child of the rows before, moved on.  The next 32
// children's starts mark their bits of the row, a lane's child is the count of
// the marks up to it: a search per item took most of the instructions of an
// item.  Called by all 32 lanes.
__device__ __forceinline__ int row_child(int u0, int nh, const TPrune* pr, int lane, int& ci) {
  const int k = ci + 1 + lane;
  const int d = k < nh ? pr->hoff[k] - u0 : 32;
  const unsigned marks = __reduce_or_sync(0xffffffffu, d < 32 ? 1u << d : 0u);
  const int c = ci + __popc(marks & (0xffffffffu >> (31 - lane)));
  ci += __popc(marks);
  return c;
}
__device__ __forceinline__ int child_shift(const TPrune* pr, int c) { return pr->rsc[pr->hch[c] >> 3]; }
__device__ __forceinline__ float3 item_pos(const TGeo& g, const float4& rel, const int4& fine, const int4& src) {
  return make_float3(fmaf((float)(fine.x + src.y), g.s_fine, rel.x), fmaf((float)(fine.y + src.z), g.s_fine, rel.y),
                     fmaf((float)(fine.z + src.w), g.s_fine, rel.z));
}

// Stages items [u0, u0 + kTCap) of the target's hit children relative to its
// cell; ci as for row_child.  Called by the whole warp.
__device__ __noinline__ int tstage_union(int u0, int total, int nh, const TPrune* pr, int lane, const TGeo& g,
                                         const float4* __restrict__ rel, const int4* __restrict__ fine, float4* spos,
                                         uint32_t* sidx, int& ci) {
  const int cnt = min(kTCap, total - u0);
#pragma unroll 1
  for (int v0 = 0; v0 < cnt; v0 += 4 * 32) {
    float4 rj[4];
    int4 fj[4], sj[4];
    uint32_t je[4];
#pragma unroll
    for (int i = 0; i < 4; ++i) {
      const int v = v0 + 32 * i;
      const int c = row_child(u0 + v, v < cnt ? nh : 0, pr, lane, ci);
      sj[i] = pr->src[c];
      const int32_t j = sj[i].x + u0 + min(v + lane, cnt - 1);
      je[i] = pack_js(j, child_shift(pr, c));
      rj[i] = rel[j];
      fj[i] = fine[j];
    }
#pragma unroll
    for (int i = 0; i < 4; ++i) {
      const int v = v0 + 32 * i + lane;
      if (v < cnt) {
        const float3 p = item_pos(g, rj[i], fj[i], sj[i]);
        spos[v] = make_float4(p.x, p.y, p.z, rj[i].w);
        sidx[v] = je[i];
      }
    }
  }
  __syncwarp();
  return cnt;
}

// Newton sums of a target at pi over all items, item u by lane u % 32, straight
// from memory: eight items' loads in flight per lane.
template <int K>
__device__ __noinline__ float2 tnewton_stream(int total, int nh, const TPrune* pr, int lane, const TGeo& g, float3 pi,
                                              float H, float Hinv, const float4* __restrict__ rel,
                                              const int4* __restrict__ fine) {
  constexpr int kB = 8;
  float Sw = 0.f, Sdw = 0.f;
  int ci = 0;
#pragma unroll 1
  for (int u0 = 0; u0 < total; u0 += kB * 32) {
    float4 rj[kB];
    int4 fj[kB], sj[kB];
#pragma unroll
    for (int i = 0; i < kB; ++i) {
      sj[i] = pr->src[row_child(u0 + 32 * i, nh, pr, lane, ci)];
      const int32_t j = sj[i].x + min(u0 + 32 * i + lane, total - 1);
      rj[i] = rel[j];
      fj[i] = fine[j];
    }
#pragma unroll
    for (int i = 0; i < kB; ++i) {
      const float3 p = item_pos(g, rj[i], fj[i], sj[i]);
      if (u0 + 32 * i + lane < total)
        tnewton_pair<K>(r2_of(pi, make_float4(p.x, p.y, p.z, 0.f)), H, Hinv, Sw, Sdw);
    }
  }
  return make_float2(Sw, Sdw);
}

// Reverse pair of target ti (support H, leaf side s_i) and source j (shift
// code sc of j seen from ti) at r^2 = r2 in ti's frame: wanted when r < H and
// r reaches past j's list radius, lowered by a margin above the rounding of r
// in either frame (the force decides again, exactly, in j's frame).  thr_j
// is j's list radius less 2^-18 of its leaf side (fine[j].w).
__device__ __forceinline__ bool want_reverse_t(float thr_j, int32_t ti, int32_t j, float r2, float H2, float H,
                                               float s_i) {
  if (!(r2 < H2) || j == ti) return false;
  const float thr = thr_j - 0x1p-18f * (s_i + H);
  return !(thr > 0.0f && r2 < thr * thr);
}
__device__ __forceinline__ bool want_reverse(const sphh::TreeDensityArgs& a, int32_t ti, int32_t j, float r2,
                                             float H2, float H, float s_i) {
  return want_reverse_t(__int_as_float(a.fine[j].w), ti, j, r2, H2, H, s_i);
}

__device__ __forceinline__ uint64_t reverse_rec(int32_t j, int32_t ti, int sc) {
  return ((uint64_t)(uint32_t)j << 32) | pack_js(ti, mirror_s(sc));
}

// Writes record k of the reverse pairs and counts it at its receiver.
__device__ __forceinline__ void emit_at(const sphh::TreeDensityArgs& a, unsigned long long k, uint64_t rec) {
  if (k < (unsigned long long)a.rev_cap) {
    a.rev_raw[k] = rec;
    atomicAdd(&a.rev_fill[(int32_t)(rec >> 32)], 1);
  } else {
    atomicOr(a.status, SPH_ST_CAPACITY);
  }
}

// Appends the reverse pairs of target ti with the marked ones of a lane's four
// sources: one counter atomic, a wait of about a microsecond, per 128 sources.
// Called by all 32 lanes.
__device__ __forceinline__ void emit_rows(const sphh::TreeDensityArgs& a, unsigned want, const uint32_t (&je)[4],
                                          int32_t ti, int lane) {
  const int mine = __popc(want);
  int incl = mine;
#pragma unroll
  for (int o = 1; o < 32; o <<= 1) {
    const int v = __shfl_up_sync(0xffffffffu, incl, o);
    if (lane >= o) incl += v;
  }
  const int all = __shfl_sync(0xffffffffu, incl, 31);
  if (all == 0) return;
  unsigned long long base = 0;
  if (lane == 0) base = atomicAdd(a.rev_count, (unsigned long long)all);
  unsigned long long k = __shfl_sync(0xffffffffu, base, 0) + (unsigned long long)(incl - mine);
#pragma unroll
  for (int i = 0; i < 4; ++i) {
    if ((want >> i) & 1u) emit_at(a, k++, reverse_rec(unpack_j(je[i]), ti, unpack_s(je[i])));
  }
}

// Appends the wanted records of the warp (one counter atomic per warp).
// Called by all 32 lanes.
__device__ __forceinline__ void emit_warp(const sphh::TreeDensityArgs& a, bool want, uint64_t rec, int lane) {
  const unsigned em = __ballot_sync(0xffffffffu, want);
  if (!em) return;
  unsigned long long base = 0;
  if (lane == 0) base = atomicAdd(a.rev_count, (unsigned long long)__popc(em));
  base = __shfl_sync(0xffffffffu, base, 0);
  if (want) {
    emit_at(a, base + (unsigned long long)__popc(em & ((1u << lane) - 1u)), rec);
  }
}

// Appends the list entries marked in each lane's mask wm (bit e: entry e of
// the lane's list): one counter atomic for the warp, then every lane writes its
// records at its offset.  Called by all 32 lanes.  (Not inlined: expanded in
// place it made the kernel 40 % longer, and instruction fetches are a part of
// its time.)
struct TEmit {
  unsigned long long* count;
  uint64_t* raw;
  int32_t* per_receiver;
  int64_t cap;
  int32_t* status;
};
__device__ __noinline__ void emit_marked(TEmit o, uint32_t wm, const TRound& S, int32_t ti, int lane) {
  const int my = __popc(wm);
  int incl = my;
#pragma unroll
  for (int d = 1; d < 32; d <<= 1) {
    const int v = __shfl_up_sync(0xffffffffu, incl, d);
    if (lane >= d) incl += v;
  }
  const int total = __shfl_sync(0xffffffffu, incl, 31);
  if (total != 0) {
    unsigned long long base = 0;
    if (lane == 0) base = atomicAdd(o.count, (unsigned long long)total);
    unsigned long long k = __shfl_sync(0xffffffffu, base, 0) + (unsigned long long)(incl - my);
#pragma unroll 1
    for (; wm != 0u; wm &= wm - 1u, ++k) {
      const uint32_t je = __float_as_uint(S.pos[S.list[__ffs((int)wm) - 1][lane]].w);
      const int32_t j = unpack_j(je);
      if (k < (unsigned long long)o.cap) {
        o.raw[k] = reverse_rec(j, ti, unpack_s(je));
        atomicAdd(&o.per_receiver[j], 1);
      } else {
        atomicOr(o.status, SPH_ST_CAPACITY);
      }
    }
  }
  __syncwarp();
}

// Outputs of target ti (source index) from its sums at h (Sec. 3.1 and the
// equation of state of Sec. 3.2).
template <int K>
__device__ __forceinline__ void tdens_write(const sphh::TreeDensityArgs& a, const PhysDev& ph, int32_t ti,
                                            float h, const TDSums& s, float u_i, int passes, bool noconv) {
  const int32_t p = a.perm[ti];
  const float H = KernT<K>::gamma * h;
  const float Hinv = 1.0f / H;
  const float H2inv = Hinv * Hinv;
  const float rho = s.mw * H2inv * Hinv;
  const float fval = 1.0f / (1.0f - s.mdw / (3.0f * s.mw));
  const float div = s.div * H2inv / s.mw;
  const float curl = sqrtf(fmaf(s.cx, s.cx, fmaf(s.cy, s.cy, s.cz * s.cz))) * H2inv / s.mw;
  const float P = (ph.gamma - 1.0f) * u_i * rho;
  const float cs = sqrtf(ph.gamma * P / rho);
  const float hf = h;
  a.h[p] = hf;
  a.rho[p] = rho;
  a.f[p] = fval;
  a.div_v[p] = div;
  a.curl_v[p] = curl;
  a.P[p] = P;
  a.c[p] = cs;
  a.B[p] = fabsf(div) / (fabsf(div) + curl + ph.eps_balsara * cs / hf);
  if (a.n_iter) a.n_iter[p] = passes;
  if (noconv) atomicOr(a.status, SPH_ST_H_NOCONV);
}

// A warp takes windows of kTWin consecutive targets from a counter: of each
// leaf the rounds (kTPer targets from the leaf's first one on) that begin in
// the window, so that a leaf's rounds, and with them the order of every sum, do
// not depend on the windows nor on what else the pool holds.
//
// Bound by instruction issue (70 % of the slots): 24 warps per SM, 1,590 warp
// instructions per particle, 3.85 ms on the 2M clustered box (7.9 when every round
// staged its ~290 sources in shared memory, 12 warps per SM, and filtered them from
// there).  The filter works on sources held in registers and keeps only the ~90
// listed ones; the loops and warp functions are not expanded in place (fetch stalls
// were the largest at 63 KB of code); windows are of two rounds, as a round beside a
// dense core tests up to 23,000 sources (with 32 targets per window the pool of 48
// uneven boxes took 1.2 times as long).
//
// kMask: the masked loops (a.act, a.act_pre set); the plain instance carries
// none of their tests.
template <int K, bool kMask>
__global__ void __launch_bounds__(kTWarps * 32, kMask ? kTMaskBlocks : kTDensBlocks)
k_tree_density(sphh::TreeDensityArgs a, PhysDev ph) {
  extern __shared__ __align__(16) unsigned char tsm[];
  const int lane = threadIdx.x & 31;
  const unsigned lt = (1u << lane) - 1u;
  // (the quartic instance is scheduled worse around constants from the parameters:
  // 96k clustered particles 1.93 -> 1.98 ms)
  const NewtonConst nwt = K == kKernQuartic
                              ? newton_const(KernT<K>::gammad, ph.eta3, ph.newton.tol, ph.newton.max_it)
                              : ph.newton;
  TRound& S = *reinterpret_cast<TRound*>(tsm + (size_t)(threadIdx.x >> 5) * kTRoundBytes);
  const int t = lane / kTreeTpp, sub = lane % kTreeTpp;
  const int32_t nl = *a.n_leaves;
  const int64_t n = a.n_total;
  unsigned long long pair_acc = 0, free_acc = 0;
  for (int64_t w0 = (int64_t)next_group(a.work, lane) * kTWin; w0 < n; w0 = (int64_t)next_group(a.work, lane) * kTWin) {
    const int32_t w1 = (int32_t)(w0 + kTWin < n ? w0 + kTWin : n);
    for (int32_t li = a.leaf_of[w0]; li < nl; ++li) {
      const TreeLeaf Lf = a.leaves[li];
      if (Lf.start >= w1) break;
      const int32_t t_hi = a.leaves[li + 1].start;
      const int32_t first =
          Lf.start >= (int32_t)w0 ? Lf.start : Lf.start + (((int32_t)w0 - Lf.start + kTPer - 1) / kTPer) * kTPer;
      if (first >= t_hi || first >= w1) continue;  // no round of this leaf begins here
      const GridDev G = a.grid[sim_of_cell(a.grid, a.n_sims, Lf.cell)];
      const TGeo g = leaf_geo(Lf, G);
      const TRanges R = load_ranges(a.ranges, li, lane);
      const int32_t cum_next = __shfl_down_sync(0xffffffffu, R.cum, 1);
      if (kMask) {
        // masked loops: a leaf without a masked particle in its 27 cells has
        // no masked target and no masked receiver of a reverse pair
        const int32_t na = lane < 27 ? a.act_pre[R.lo + (cum_next - R.cum)] - a.act_pre[R.lo] : 0;
        if (!__any_sync(0xffffffffu, na > 0)) continue;
      }
      const float hcap = h_cap_depth(G, Lf.depth);
      // few sources: the 27 ranges whole; else the children of the ranges
      // that some target of the round reaches (children are half the cell; a
      // cell at the deepest level has one child)
      const bool whole = R.nsrc <= kTWhole;
      const bool shifted = __any_sync(0xffffffffu, R.sc != kNoShift);
      const float cside = Lf.depth < kTreeDepth ? 0.5f * g.side : g.side;
      uint32_t cand_all = 0, cand_act = 0;
      int nseg = 0, total = 0;
      if (whole) {
        __syncwarp();
        const bool some = lane < 27 && cum_next > R.cum;
        const unsigned bm = __ballot_sync(0xffffffffu, some);
        if (some) S.seg[__popc(bm & lt)] = make_int2(R.cum, (int)pack_js(R.lo, R.sc));
        nseg = __popc(bm);
        total = R.nsrc;
        __syncwarp();
      } else {
        prune_tables(a.skey, R, Lf.depth, lane, &S.tab, kMask ? a.act_pre : nullptr);
        cand_all = group_candidates(sub, &S.tab, false);
        if (kMask) cand_act = group_candidates(sub, &S.tab, true);
      }
#pragma unroll 1
      for (int32_t t0 = first; t0 < t_hi && t0 < w1; t0 += kTPer) {
        const bool valid = t0 + t < t_hi;
        const int32_t ti = a.tgt[t0 + (valid ? t : 0)];
        // masked loops: a target outside the mask keeps its h and outputs; its
        // list, of masked sources, only sends reverse pairs to them (their
        // forces need every pair within either support)
        const bool on = valid && (!kMask || a.act[ti] != 0);
        const float4 reli = a.rel[ti];
        const int4 fi = a.fine[ti];
        const float3 pi = rel_to(g, reli, fi, kNoShift);
        const float4 vi = a.vel4[ti];
        const float Ri = a.lrad[ti];
        const float R2 = Ri * Ri;
        const float h_start = a.hs[ti];
        __syncwarp();  // the previous round is done with the shared arrays
        if (sub == 0) S.tgt[t] = make_float4(pi.x, pi.y, pi.z, valid ? R2 : -1.0f);
        if (!whole) {
          const int2 st = prune_round_fast(valid, sub, lane, pi, R2 * (1.0f + 0x1p-10f), g.side, cside, &S.tab,
                                           !kMask || on ? cand_all : cand_act, S.seg);
          nseg = st.x;
          total = st.y;
        }
        __syncwarp();
        // masked loops: which targets are in the mask (bit 8 q: target q)
        const unsigned on_mask = kMask ? __ballot_sync(0xffffffffu, on) : 0xffffffffu;
        int nq = 0;  // the sources the lane's target lists, once more were kept than fit
#pragma unroll 1
        for (unsigned todo = (1u << kTPer) - 1u; todo != 0u;) {
          // the round's targets, or as many of them as are known to fit
          unsigned now = 0u;
          for (int q = 0, sum = 0; q < kTPer; ++q) {
            sum += ((todo >> q) & 1u) ? __shfl_sync(0xffffffffu, nq, q * kTreeTpp) : 0;
            if (((todo >> q) & 1u) && (now == 0u || sum <= kTKept)) now |= 1u << q;
          }
          // 1. filter: the sources 32 at a time, one per lane; the round's
          // targets test each in turn.  Those within some target's list radius
          // are kept; lane sub of a target lists the kept slots of its own
          // sources, every kTreeTpp-th of the segments' sequence, in order.
          // A target whose list overflows (it leaves for the per-target kernel)
          // stops listing, so that a round beside a dense core does not go on
          // collecting the core.
          unsigned live = now;
          int cnt = 0, kept = 0, seg0 = 0;
#pragma unroll 1
          for (int u0 = 0; u0 < total; u0 += 64) {
            const unsigned over = __ballot_sync(0xffffffffu, cnt > kTreeList);
            if (over != 0u) {
#pragma unroll
              for (int q = 0; q < kTPer; ++q)
                if ((over >> (q * kTreeTpp)) & kTGroup) live &= ~(1u << q);
              if (live == 0u) break;
            }
            float4 rj[2];
            int4 fj[2];
            uint32_t je[2];
            bool aj[2];
#pragma unroll
            for (int i = 0; i < 2; ++i) {
              // the segment of source u: the starts that fall into these 32
              // sources, as a bit mask, count up to lane
              const int ub = u0 + 32 * i, u = ub + lane, s = seg0 + 1 + lane;
              const int st = s < nseg ? S.seg[s].x - ub : 32;
              const unsigned bits = __reduce_or_sync(0xffffffffu, st < 32 ? 1u << st : 0u);
              const int2 sg = S.seg[seg0 + __popc(bits & (lt | (1u << lane)))];
              seg0 += __popc(bits);
              je[i] = (uint32_t)sg.y + (uint32_t)(u - sg.x);
              const int32_t j = u < total ? unpack_j(je[i]) : ti;
              rj[i] = a.rel[j];
              fj[i] = a.fine[j];
              aj[i] = kMask ? a.act[j] != 0 : true;
            }
#pragma unroll
            for (int i = 0; i < 2; ++i) {
              const float3 p = shifted ? rel_to(g, rj[i], fj[i], unpack_s(je[i])) : rel_to(g, rj[i], fj[i], kNoShift);
              const bool in = u0 + 32 * i + lane < total;
              unsigned any = 0u, own = 0u;
#pragma unroll
              for (int q = 0; q < kTPer; ++q) {
                const float4 T = S.tgt[q];
                // (a target outside the mask lists the masked sources only)
                const bool is = in && r2_of(make_float3(T.x, T.y, T.z), make_float4(p.x, p.y, p.z, 0.f)) < T.w &&
                                (!kMask || aj[i] || ((on_mask >> (q * kTreeTpp)) & 1u));
                const unsigned hit = ((live >> q) & 1u) ? __ballot_sync(0xffffffffu, is) : 0u;
                any |= hit;
                if (q == t) own = hit;
              }
              if ((any >> lane) & 1u) {
                const int at = kept + __popc(any & lt);
                if (at < kTKept) S.pos[at] = make_float4(p.x, p.y, p.z, __uint_as_float(je[i]));
              }
#pragma unroll 1
              for (unsigned m = (own >> sub) & kTLanes; m != 0u; m &= m - 1u) {
                const int b = __ffs((int)m) - 1 + sub;
                S.list[min(cnt, kTreeList)][lane] = (uint8_t)(kept + __popc(any & ((1u << b) - 1u)));
                ++cnt;
              }
              kept += __popc(any);
            }
          }
          __syncwarp();
          if (kept > kTKept && live != 0u && (live != now || (live & (live - 1u)) != 0u)) {
            // too many sources are near some target: fewer targets at a time
            // (one target's list of up to kTreeTpp * kTreeList sources fits);
            // those that left are done
            const int nt = gsumi(cnt);
            if ((now >> t) & 1u) nq = nt;
            now &= ~live;
          }
          if (now == 0u) continue;
          todo &= ~now;
          const bool act_now = valid && ((now >> t) & 1u), on_now = act_now && on;
          // a target whose list overflowed, or whose support outgrows R_i, leaves
          // the round: it is queued for the per-target kernel, which solves it at
          // its own level with all 32 lanes of a warp over its 27 cells (so the
          // other targets of its round do not wait for it).  The flag is shared
          // by the target's lanes.
          bool queued = group_any(cnt > kTreeList, lane);
          // 2. Newton-Raphson passes
          float h = valid ? h_start : hcap;
          if (on) {
            if (!(h > 0.0f)) h = 0.5f * hcap;
            if (h > hcap) h = hcap;
          }
          if (valid && KernT<K>::gamma * h > Ri) queued = true;
          float hlo = 0.0f, hhi = INFINITY;
          bool done = !on_now || queued, atcap = false, conv = false;
          int it = 0, passes = 0;
#pragma unroll 1
          while (__any_sync(0xffffffffu, !done)) {
            const float H = KernT<K>::gamma * h;
            const float Hinv = 1.0f / H;
            float Sw = 0.f, Sdw = 0.f;
            if (!done)
#pragma unroll 1
              for (int e = 0; e < cnt; ++e) tnewton_pair<K>(r2_of(pi, S.pos[S.list[e][lane]]), H, Hinv, Sw, Sdw);
            Sw = gsum(Sw);
            Sdw = gsum(Sdw);
            if (!done) {
              passes = it + 1;
              if (newton_update(Sw, Sdw, nwt, hcap, h, hlo, hhi, it, atcap, conv)) done = true;
            }
            // the list holds r < R_i: a support beyond it is queued
            if (act_now && !queued && !atcap && KernT<K>::gamma * h > Ri) {
              queued = true;
              done = true;
            }
          }
          // 3. final pass at h; the list's reverse pairs are marked on the way
          // (bit e: entry e), with j's threshold read with its fine position.
          // The list is published for the force loop as it is walked: entry e of
          // every lane, lane by lane, then entry e + 1, close to the sources'
          // order, so that the lanes of the force's targets read neighbouring
          // sources
          const float H = KernT<K>::gamma * h;
          const float Hinv = 1.0f / H;
          const float H2 = H * H;
          TDSums s;
          tds_zero(s);
          uint32_t wm = 0;
          const int mine = on_now && !queued ? cnt : 0;
          uint32_t* dst = a.lists + (int64_t)ti * kTreeListTarget;
          int all = 0;
#pragma unroll 1
          for (int e = 0;; ++e) {
            const unsigned m = __ballot_sync(0xffffffffu, e < mine);
            if (m == 0u) break;
            const unsigned row = (m >> (t * kTreeTpp)) & kTGroup;
            if (e < mine) {
              const float4 pk = S.pos[S.list[e][lane]];
              const uint32_t je = __float_as_uint(pk.w);
              const int32_t j = unpack_j(je);
              dst[all + __popc(row & ((1u << sub) - 1u))] = je;
              const float4 rj = a.rel[j];
              const int4 fj = a.fine[j];
              const float3 d = pair_vec(g, reli, fi, rj, fj, unpack_s(je));
              tdens_pair<K>(d.x, d.y, d.z, vi, a.vel4[j], rj.w, H, Hinv, s);
              if (!atcap && want_reverse_t(__int_as_float(fj.w), ti, j, r2_of(pi, pk), H2, H, g.side) &&
                  (!kMask || a.act[j] != 0))
                wm |= 1u << e;
            }
            all += __popc(row);
          }
          if (on_now && sub == 0) a.list_cnt[ti] = (uint16_t)(atcap || queued ? kListFallback : all);
          if (kMask && act_now && !queued && !on) {
            // outside the mask: the reverse pairs to its listed (masked) sources
#pragma unroll 1
            for (int e = 0; e < cnt; ++e) {
              const float4 pk = S.pos[S.list[e][lane]];
              if (want_reverse(a, ti, unpack_j(__float_as_uint(pk.w)), r2_of(pi, pk), H2, H, g.side)) wm |= 1u << e;
            }
          }
          // reverse pairs from the lists: the warp takes one slot range for the
          // whole round
          emit_marked(TEmit{a.rev_count, a.rev_raw, a.rev_fill, a.rev_cap, a.status}, wm, S, ti, lane);
          tcombine(s);
          if (act_now && sub == 0) {
            if (queued) {
              // solved at its own level by the per-target kernel
              const int32_t k = atomicAdd(a.fb_count, 1);
              if (k < a.n_total) a.fb_list[k] = ti | kFbOwnLevel | (on ? 0 : kFbPassive);
              free_acc += on ? 1ull : 0ull;
            } else if (on) {
              tdens_write<K>(a, ph, ti, h, s, vi.w, passes, !conv && !atcap);
              if (atcap) {
                // the support outgrew this level: re-solved at a coarser one
                const int32_t k = atomicAdd(a.fb_count, 1);
                if (k < a.n_total) a.fb_list[k] = ti;
              } else {
                pair_acc += (unsigned long long)s.npair;
              }
            }
          }
          __syncwarp();
        }
      }
    }
  }
  if (ph.count_pairs) {
    unsigned long long v = pair_acc, w = free_acc;
#pragma unroll
    for (int o = 16; o > 0; o >>= 1) {
      v += __shfl_xor_sync(0xffffffffu, v, o);
      w += __shfl_xor_sync(0xffffffffu, w, o);
    }
    if (lane == 0 && v) atomicAdd(a.pairs, v);
    if (lane == 0 && w) atomicAdd(a.list_free, w);
  }
}

// Reverse pairs -> per-receiver segments: rev_start holds the exclusive scan
// of the counts; each pair takes a slot of its receiver's segment.
__global__ void k_rev_scatter(const uint64_t* __restrict__ raw, const unsigned long long* __restrict__ count,
                              int64_t cap, const int32_t* __restrict__ start, int32_t* __restrict__ fill,
                              uint32_t* __restrict__ rev) {
  const int64_t m = (int64_t)min(*count, (unsigned long long)cap);
  for (int64_t k = (int64_t)blockIdx.x * blockDim.x + threadIdx.x; k < m; k += (int64_t)gridDim.x * blockDim.x) {
    const uint64_t e = raw[k];
    const int32_t r = (int32_t)(e >> 32);
    const int32_t pos = start[r] + atomicAdd(&fill[r], 1);
    rev[pos] = (uint32_t)(e & 0xffffffffu);
  }
}

// A segment of at most N entries sorted in registers: a bitonic network
// (every index fixed at compile time), padded with the largest key.
template <int N>
__device__ __forceinline__ void sort_segment_regs(uint32_t* rev, int32_t len) {
  uint32_t v[N];
#pragma unroll
  for (int k = 0; k < N; ++k) v[k] = k < len ? rev[k] : 0xffffffffu;
#pragma unroll
  for (int k = 2; k <= N; k <<= 1) {
#pragma unroll
    for (int j = k >> 1; j > 0; j >>= 1) {
#pragma unroll
      for (int i = 0; i < N; ++i) {
        const int l = i ^ j;
        if (l > i) {
          const uint32_t x = v[i], y = v[l];
          const bool up = (i & k) == 0;
          v[i] = up ? min(x, y) : max(x, y);
          v[l] = up ? max(x, y) : min(x, y);
        }
      }
    }
  }
#pragma unroll
  for (int k = 0; k < N; ++k)
    if (k < len) rev[k] = v[k];
}

// Sorts each receiver's segment by packed source (the slot order above is
// arbitrary), so the force sums run in a fixed order.  A block's receivers own
// one contiguous run of entries: it passes through shared memory when it fits,
// so that memory sees whole sectors (138 -> 103 us for the 17.7M entries of
// the 2M clustered box).  Segments of up to 32 are sorted by a thread in
// registers; longer ones are queued for k_rev_mid (from the queue's front) and
// k_rev_long (from its back).
constexpr int kRevThreads = 256;
constexpr int kRevBuf = 6144;
constexpr int kRevShort = 32;
constexpr int kRevMid = 512;
__global__ void __launch_bounds__(kRevThreads)
k_rev_sort(int64_t n, const int32_t* __restrict__ start, uint32_t* __restrict__ rev, int32_t* __restrict__ queue,
           int32_t* __restrict__ n_mid, int32_t* __restrict__ n_long) {
  __shared__ uint32_t buf[kRevBuf];
  for (int64_t i0 = (int64_t)blockIdx.x * kRevThreads; i0 < n; i0 += (int64_t)gridDim.x * kRevThreads) {
    const int64_t i1 = i0 + kRevThreads < n ? i0 + kRevThreads : n;
    const int32_t e0 = start[i0], m = start[i1] - e0;
    const bool staged = m <= kRevBuf;
    if (staged) {
      for (int32_t k = threadIdx.x; k < m; k += kRevThreads) buf[k] = rev[e0 + k];
      __syncthreads();
    }
    const int64_t i = i0 + threadIdx.x;
    if (i < i1) {
      const int32_t b = start[i], len = start[i + 1] - b;
      uint32_t* seg = staged ? buf + (b - e0) : rev + b;
      if (len > kRevMid)
        queue[n - 1 - atomicAdd(n_long, 1)] = (int32_t)i;
      else if (len > kRevShort)
        queue[atomicAdd(n_mid, 1)] = (int32_t)i;
      else if (len > 16)
        sort_segment_regs<32>(seg, len);
      else if (len > 8)
        sort_segment_regs<16>(seg, len);
      else if (len > 1)
        sort_segment_regs<8>(seg, len);
    }
    if (staged) {
      __syncthreads();
      for (int32_t k = threadIdx.x; k < m; k += kRevThreads) rev[e0 + k] = buf[k];
      __syncthreads();
    }
  }
}

// Bitonic sort of len > 1 entries by `threads` threads (index me), sync() between
// the steps.  Its compare-exchanges all put the smaller entry first (each merge
// opens with mirrored partners), so that entries past the end need no padding.
template <class Sync>
__device__ __forceinline__ void sort_segment(uint32_t* seg, int32_t len, int me, int threads, Sync sync) {
  int32_t half = 1;  // pairs of a step: half the padded length
  while (2 * half < len) half <<= 1;
#pragma unroll 1
  for (int32_t k = 1; k <= half; k <<= 1) {
#pragma unroll 1
    for (int32_t j = k; j > 0; j >>= 1) {
#pragma unroll 1
      for (int32_t p = me; p < half; p += threads) {
        const int32_t lo = ((p & ~(j - 1)) << 1) | (p & (j - 1));
        const int32_t hi = j == k ? (lo ^ (2 * k - 1)) : lo + j;
        if (hi < len) {
          const uint32_t x = seg[lo], y = seg[hi];
          if (x > y) {
            seg[lo] = y;
            seg[hi] = x;
          }
        }
      }
      sync();
    }
  }
}

// A segment of at most 32 R entries sorted by a warp, lane l's registers holding
// places l R .. l R + R - 1: the bitonic network with strides below R within a
// lane and the others by shuffles, padded with the largest key.  (Up to 256
// entries so, against the network in shared memory: the pool of 48 boxes 99 -> 40
// us, 300k particles with Wendland C2 46 -> 22.)
template <int R>
__device__ __forceinline__ void sort_segment_warp(uint32_t* seg, int32_t len, int lane) {
  uint32_t v[R];
#pragma unroll
  for (int r = 0; r < R; ++r) v[r] = 32 * r + lane < len ? seg[32 * r + lane] : 0xffffffffu;  // (any order)
  __syncwarp();
#pragma unroll
  for (int k = 2; k <= 32 * R; k <<= 1) {
#pragma unroll
    for (int j = k >> 1; j > 0; j >>= 1) {
#pragma unroll
      for (int r = 0; r < R; ++r) {
        const bool up = ((lane * R + r) & k) == 0;
        if (j >= R) {
          const uint32_t o = __shfl_xor_sync(0xffffffffu, v[r], j / R);
          v[r] = (((lane * R) & j) == 0) == up ? min(v[r], o) : max(v[r], o);
        } else if ((r & j) == 0) {
          const uint32_t x = v[r], y = v[r | j];
          v[r] = up ? min(x, y) : max(x, y);
          v[r | j] = up ? max(x, y) : min(x, y);
        }
      }
    }
  }
#pragma unroll
  for (int r = 0; r < R; ++r)
    if (lane * R + r < len) seg[lane * R + r] = v[r];
}

// The queued segments: up to kRevMid entries a warp each, longer ones a block
// each (in place in global memory beyond its buffer).  A thread's insertion sort
// of them took 0.8 of the 3.4 ms of the pool of 48 uneven boxes, whose dense
// cores receive from hundreds of larger supports.
__global__ void __launch_bounds__(kRevThreads)
k_rev_mid(const int32_t* __restrict__ start, uint32_t* __restrict__ rev, const int32_t* __restrict__ queue,
          const int32_t* __restrict__ n_mid) {
  __shared__ uint32_t buf[kRevThreads / 32][kRevMid];
  const int warp = threadIdx.x >> 5, lane = threadIdx.x & 31;
  const int32_t nq = *n_mid, warps = gridDim.x * (kRevThreads / 32);
  for (int32_t q = blockIdx.x * (kRevThreads / 32) + warp; q < nq; q += warps) {
    const int32_t i = queue[q], b = start[i], len = start[i + 1] - b;
    if (len <= 64) {
      sort_segment_warp<2>(rev + b, len, lane);
      continue;
    }
    if (len <= 128) {
      sort_segment_warp<4>(rev + b, len, lane);
      continue;
    }
    if (len <= 256) {
      sort_segment_warp<8>(rev + b, len, lane);
      continue;
    }
    for (int32_t k = lane; k < len; k += 32) buf[warp][k] = rev[b + k];
    __syncwarp();
    sort_segment(buf[warp], len, lane, 32, [] { __syncwarp(); });
    for (int32_t k = lane; k < len; k += 32) rev[b + k] = buf[warp][k];
    __syncwarp();
  }
}

__global__ void __launch_bounds__(kRevThreads)
k_rev_long(int64_t n, const int32_t* __restrict__ start, uint32_t* __restrict__ rev, const int32_t* __restrict__ queue,
           const int32_t* __restrict__ n_long) {
  __shared__ uint32_t buf[kRevBuf];
  const int32_t nq = *n_long;
  for (int32_t q = blockIdx.x; q < nq; q += gridDim.x) {
    const int32_t i = queue[n - 1 - q], b = start[i], len = start[i + 1] - b;
    const bool staged = len <= kRevBuf;
    if (staged)
      for (int32_t k = threadIdx.x; k < len; k += kRevThreads) buf[k] = rev[b + k];
    __syncthreads();
    sort_segment(staged ? buf : rev + b, len, threadIdx.x, kRevThreads, [] { __syncthreads(); });
    if (staged)
      for (int32_t k = threadIdx.x; k < len; k += kRevThreads) rev[b + k] = buf[k];
    __syncthreads();
  }
}

// ---- force ------------------------------------------------------------------

struct TFSums {
  float ax, ay, az, du, vsig;
  int npair;
};

// A source's force record, in source order (written by the force gather): q0 =
// (rel x, y, z, H), q1 = (fine x, y, z, rho as bits), q2 = (v, m), q3 =
// (f P / rho^2, f, c, B), each in an array of its own: a target's eight lanes
// read neighbouring sources, whose quarters share a line or two.  With 64-byte
// records and lists in the density lanes' order the force gathers filled the L1's
// data stage (94 % of its wavefronts): 2M clustered particles 1306 -> 1023 us.
// 1/H is recomputed (correctly rounded, the value the arrays held).
struct TRec {
  float4 q0;
  int4 q1;
};

__device__ __forceinline__ TRec trec_head(const sphh::TreeForceArgs& a, int32_t j) {
  TRec t;
  t.q0 = a.rec[j];
  t.q1 = *reinterpret_cast<const int4*>(a.rec + a.n_total + j);
  return t;
}
__device__ __forceinline__ float4 trec_vel(const sphh::TreeForceArgs& a, int32_t j) { return a.rec[2 * a.n_total + j]; }
__device__ __forceinline__ float4 trec_pres(const sphh::TreeForceArgs& a, int32_t j) { return a.rec[3 * a.n_total + j]; }

// Flavours of the force kernels: the "Minimal" force, the SPHENIX force and
// the SPHENIX gradient pass (Sec. 3.3; the terms are those of force.cu's
// flavours, with the fifth record E = (u, alpha_V, P, alpha_c) per source).
// The time-step limiter (kTLimit, Sec. 3.4) and the wake-up pass (kTWake)
// walk the same pairs with fE.x = each source's time bin.
enum : int { kTMin = 0, kTSphenix = 1, kTGradient = 2, kTLimit = 3, kTWake = 4 };

// One force pair with x_ij = (dx, dy, dz) (same terms as force.cu).  The
// gradient pass keeps only r < H_i (G_i = 0 beyond): the Laplacian sum
// (m_j / rho_j)(u_i - u_j) G_i in ax, the largest alpha_V in ay and the
// largest conduction speed v_c,ij in vsig.
template <int kFl, int K>
__device__ __forceinline__ void tforce_pair(float dx, float dy, float dz, const float4& vi, const float4& ci,
                                            const float4& ei, float Hi, float Hinv_i, float rho_i, const float4& vj,
                                            const float4& cj, const float4& ej, float Hj, float Hinv_j,
                                            float rho_j, const PhysDev& ph, TFSums& s) {
  const float r2 = fmaf(dx, dx, fmaf(dy, dy, dz * dz));
  if constexpr (kFl == kTLimit) {
    // the largest bin among the force pairs (r < max(H_i, H_j)) in vsig
    const float Hm = fmaxf(Hi, Hj);
    const bool in = r2 < Hm * Hm;
    s.vsig = in ? fmaxf(s.vsig, ej.x) : s.vsig;
    s.npair += in;
    return;
  }
  const float rinv = rsqrt_norm(fmaxf(r2, 1e-30f));
  const float r = r2 * rinv;
  const float hi2 = Hinv_i * Hinv_i;
  const float Gi = kernel_g<K>(r * Hinv_i, Hi * rinv) * (hi2 * hi2 * Hinv_i);
  const float vx = vi.x - vj.x, vy = vi.y - vj.y, vz = vi.z - vj.z;
  const float vdotx = fmaf(vx, dx, fmaf(vy, dy, vz * dz));
  if constexpr (kFl == kTGradient) {
    s.ax = fmaf(div_norm(vj.w, rho_j) * (ei.x - ej.x), Gi, s.ax);
    const float vc = fmaf(fabsf(vdotx), rinv, sqrtf(div_norm(2.0f * fabsf(ei.z - ej.z), rho_i + rho_j)));
    const bool in = r2 < Hi * Hi;
    s.vsig = in ? fmaxf(s.vsig, vc) : s.vsig;
    s.ay = in ? fmaxf(s.ay, ej.y) : s.ay;
    s.npair += in;
    return;
  }
  const float hj2 = Hinv_j * Hinv_j;
  const float Gj = kernel_g<K>(r * Hinv_j, Hj * rinv) * (hj2 * hj2 * Hinv_j);
  const float mu = fminf(vdotx, 0.0f) * rinv;
  const float vs = fmaf(-ph.beta_v, mu, ci.z + cj.z);
  const float av = kFl == kTSphenix ? 0.5f * (ei.y + ej.y) : ph.alpha_v;
  const float nu = div_norm(-av * (ci.w + cj.w) * mu * vs, rho_i + rho_j);
  const float piG = ci.x * Gi;
  const float visc = fmaf(ci.y, Gi, cj.y * Gj);
  const float mj = vj.w;
  const float sc = mj * fmaf(0.5f * nu, visc, fmaf(cj.x, Gj, piG));
  s.ax = fmaf(-sc, dx, s.ax);
  s.ay = fmaf(-sc, dy, s.ay);
  s.az = fmaf(-sc, dz, s.az);
  s.du = fmaf(mj * fmaf(0.25f * nu, visc, piG), vdotx, s.du);
  if constexpr (kFl == kTSphenix) {
    // conduction: zero beyond both supports (visc = 0) and for r = 0
    const float Ps = ei.z + ej.z, rs = rho_i + rho_j;
    const float ac = Ps > 0.0f ? __fdividef(fmaf(ei.z, ei.w, ej.z * ej.w), Ps) : 0.0f;
    const float vc = fmaf(fabsf(vdotx), rinv, sqrtf(div_norm(2.0f * fabsf(ei.z - ej.z), rs)));
    s.du = fmaf(mj * ac * vc * (ei.x - ej.x) * r, div_norm(visc, rs), s.du);
  }
  const float Hm = fmaxf(Hi, Hj);
  const bool in = r2 < Hm * Hm;
  s.vsig = in ? fmaxf(s.vsig, vs) : s.vsig;
  s.npair += in;
}

// tforce_pair with source j's data from its record (head already loaded) and,
// for the flavours with one, its fifth record.  The wake-up pass raises the
// wake-up bin of a source outside the mask within r < max(H_i, H_j) whose bin
// lies below the target's bin - 2 (Saitoh & Makino's limiter, Sec. 3.4).
template <int kFl, int K>
__device__ __forceinline__ void tforce_rec(float dx, float dy, float dz, const float4& vi, const float4& ci,
                                           const float4& ei, float Hi, float Hinv_i, float rho_i,
                                           const sphh::TreeForceArgs& a, int32_t j, const TRec& h, const PhysDev& ph,
                                           TFSums& s) {
  if constexpr (kFl == kTWake) {
    const float r2 = fmaf(dx, dx, fmaf(dy, dy, dz * dz));
    const float Hm = fmaxf(Hi, h.q0.w);
    const int w = (int)ei.x - 2;
    if (r2 < Hm * Hm && a.act[j] == 0 && w > (int)a.fE[j].x) atomicMax(a.wake + a.perm[j], w);
    return;
  }
  const float4 ej = kFl != kTMin ? a.fE[j] : make_float4(0.f, 0.f, 0.f, 0.f);
  if constexpr (kFl == kTLimit) {
    tforce_pair<kFl, K>(dx, dy, dz, vi, ci, ei, Hi, Hinv_i, rho_i, vi, ci, ej, h.q0.w, 0.0f, 0.0f, ph, s);
  } else {
    tforce_pair<kFl, K>(dx, dy, dz, vi, ci, ei, Hi, Hinv_i, rho_i, trec_vel(a, j), trec_pres(a, j), ej, h.q0.w, __frcp_rn(h.q0.w),
                        __int_as_float(h.q1.w), ph, s);
  }
}

// The result of a target: the force, or the gradient pass's conduction
// parameter (the Euler step of eq. "artconddt" and its limiters, as in
// force.cu) and Laplacian.
template <int kFl>
__device__ __forceinline__ void tforce_write(const sphh::TreeForceArgs& a, const SphenixDev& x, float dt,
                                             int32_t ti, float Hi, const float4& ei, const TFSums& s) {
  const int32_t p = a.perm[ti];
  if constexpr (kFl == kTLimit) {
    // a step at most 4 times the smallest neighbour step: at most two bins
    // below the largest neighbour bin
    const int own = (int)ei.x, nb = (int)s.vsig - 2;
    a.bins_out[p] = own > nb ? own : nb;
  } else if constexpr (kFl == kTWake) {
    // the wake-up pass writes per source
  } else if constexpr (kFl == kTGradient) {
    const float lap = 2.0f * s.ax;
    const float src = ei.x > 0.0f ? x.beta_c * Hi * lap / sqrtf(ei.x) : 0.0f;
    const float rate = src - (ei.w - x.ac_min) * s.vsig / Hi;
    float an = fmaf(dt, rate, ei.w);
    an = fminf(an, x.ac_max * (1.0f - s.ay / x.av_max));
    an = fmaxf(an, x.ac_min);
    a.alpha_c_out[p] = an;
    if (a.lap_u != nullptr) a.lap_u[p] = lap;
  } else {
    a.ax[p] = s.ax;
    a.ay[p] = s.ay;
    a.az[p] = s.az;
    a.du_dt[p] = s.du;
    a.v_sig[p] = s.vsig;
  }
}

__device__ __forceinline__ float3 rec_rel_to(const TGeo& g, const TRec& h, int sc) {
  return rel_to(g, h.q0, h.q1, sc);
}

// A warp takes windows of win consecutive targets from a counter, kTPer at a
// time with kTreeTpp lanes each, whatever their leaves (a target's lanes hold
// its own leaf's corner): every round is full, and a large leaf is shared by
// many warps.  Bound by the L1 wavefronts of the record gathers (79 %) and by
// instruction issue (61 %).
template <int kFl, int K>
__global__ void __launch_bounds__(kTWarps * 32) k_tree_force(sphh::TreeForceArgs a, PhysDev ph, SphenixDev x,
                                                             int win) {
  const int lane = threadIdx.x & 31;
  const int t = lane / kTreeTpp, sub = lane % kTreeTpp;
  const int64_t n = a.n_total;
  unsigned long long pair_acc = 0;
  for (int64_t w0 = (int64_t)next_group(a.work, lane) * win; w0 < n;
       w0 = (int64_t)next_group(a.work, lane) * win) {
#pragma unroll 1
    for (int64_t t0 = w0; t0 < w0 + win && t0 < n; t0 += kTPer) {
      const bool valid = t0 + t < n;
      const int64_t k = t0 + (valid ? t : 0);
      const int32_t ti = a.tgt[k];
      // masked loops: skip a round without a masked target
      if (a.act != nullptr && !__any_sync(0xffffffffu, a.act[ti] != 0)) continue;
      const TreeLeaf Lf = a.leaves[a.leaf_of[k]];
      const int sim = sim_of_cell(a.grid, a.n_sims, Lf.cell);
      const TGeo g = leaf_geo(Lf, a.grid[sim]);
      const float dt = kFl == kTGradient ? (float)(x.dt_dev != nullptr ? x.dt_dev[sim] : x.dt) : 0.0f;
      TFSums s;
      s.ax = s.ay = s.az = s.du = s.vsig = 0.f;
      s.npair = 0;
      const int lc = (int)a.list_cnt[ti];   // the target's packed list
      const bool fb = lc == kListFallback;  // written by k_tree_force_fb
      const float4 ei = kFl != kTMin ? a.fE[ti] : make_float4(0.f, 0.f, 0.f, 0.f);
      if (kFl == kTGradient) s.ay = ei.y;  // alpha_V,max starts at the target's
      const TRec hi = trec_head(a, ti);
      const float Hi = hi.q0.w;
      const bool on = valid && !fb && (a.act == nullptr || a.act[ti] != 0);
      if (on) {
        const float4 reli = hi.q0;
        const int4 fi = hi.q1;
        const float3 pi = rel_to(g, reli, fi, kNoShift);
        const float4 vi = trec_vel(a, ti);
        const float4 ci = trec_pres(a, ti);
        const float2 di = make_float2(__int_as_float(hi.q1.w), __frcp_rn(hi.q0.w));
        // own reach: the list radius (a target without a complete list went
        // to the per-target kernel, kListFallback)
        const float C = a.lrad[ti];
        const float C2 = C * C;
        const uint32_t* lst = a.lists + (int64_t)ti * kTreeListTarget;
        for (int e = sub; e < lc; e += kTreeTpp) {
          const uint32_t je = lst[e];
          const int32_t j = unpack_j(je);
          if (j == ti) continue;
          const TRec hj = trec_head(a, j);
          const float3 d = pair_vec(g, reli, fi, hj.q0, hj.q1, unpack_s(je));
          tforce_rec<kFl, K>(d.x, d.y, d.z, vi, ci, ei, Hi, di.y, di.x, a, j, hj, ph, s);
        }
        // reverse pairs beyond the own reach, split between the lanes (the
        // gradient pass reaches only H_i <= the own reach: none of them)
        if (kFl != kTGradient) {
          const int32_t r0 = a.rev_start[ti], r1 = a.rev_start[ti + 1];
          for (int32_t k = r0 + sub; k < r1; k += kTreeTpp) {
            const uint32_t je = a.rev[k];
            const int32_t j = unpack_j(je);
            const TRec hj = trec_head(a, j);
            const float3 pj = rec_rel_to(g, hj, unpack_s(je));
            const float dx = pi.x - pj.x, dy = pi.y - pj.y, dz = pi.z - pj.z;
            if (fmaf(dx, dx, fmaf(dy, dy, dz * dz)) >= C2)
              tforce_rec<kFl, K>(dx, dy, dz, vi, ci, ei, Hi, di.y, di.x, a, j, hj, ph, s);
          }
        }
      }
      s.ax = gsum(s.ax);
      s.ay = kFl == kTGradient ? gmax(s.ay) : gsum(s.ay);
      s.az = gsum(s.az);
      s.du = gsum(s.du);
      s.vsig = gmax(s.vsig);
      s.npair = gsumi(s.npair);
      if (on && sub == 0) {
        tforce_write<kFl>(a, x, dt, ti, Hi, ei, s);
        pair_acc += (unsigned long long)s.npair;
      }
    }
  }
  if (ph.count_pairs && a.pairs != nullptr) {
    unsigned long long v = pair_acc;
#pragma unroll
    for (int o = 16; o > 0; o >>= 1) v += __shfl_xor_sync(0xffffffffu, v, o);
    if (lane == 0 && v) atomicAdd(a.pairs, v);
  }
}

// ---- fallback: targets whose support outgrew the cells of their level ------
//
// One warp per queued target, all 32 lanes over its candidates: the 27 cells
// one level coarser (twice the side) around it, then coarser still while the
// solve keeps hitting the cap.  A target that needs more than its top cell
// sets SPH_ST_REBUILD: the top grid itself is too fine.

__device__ __forceinline__ float wsum(float v) {
#pragma unroll
  for (int o = 16; o > 0; o >>= 1) v += __shfl_xor_sync(0xffffffffu, v, o);
  return v;
}

__device__ __forceinline__ int wsumi(int v) {
#pragma unroll
  for (int o = 16; o > 0; o >>= 1) v += __shfl_xor_sync(0xffffffffu, v, o);
  return v;
}

// The 27 ranges of cell L (lanes 0..26) as a TRanges record.
__device__ __forceinline__ TRanges cell_ranges(const GridDev& G, const TreeLeaf& L,
                                               const uint64_t* __restrict__ skey,
                                               const int32_t* __restrict__ cell_start, int lane) {
  TRanges R;
  int32_t len = 0;
  R.lo = 0;
  R.sc = kNoShift;
  if (lane < 27) {
    const TreeRange t = neighbour_range(G, L, lane, skey, cell_start);
    R.lo = t.lo;
    len = t.hi - t.lo;
    R.sc = t.shift;
  }
  int incl = len;
#pragma unroll
  for (int o = 1; o < 32; o <<= 1) {
    const int v = __shfl_up_sync(0xffffffffu, incl, o);
    if (lane >= o) incl += v;
  }
  R.cum = incl - len;
  R.nsrc = __shfl_sync(0xffffffffu, incl, 31);
  return R;
}

// The targets that left their round, a warp each: mostly low-density targets
// beside a dense core, whose 27 cells hold thousands of sources.  There are few
// of them (4040 of 690k particles in a pool of 48 boxes), so the kernel lasts
// about as long as its largest target: what counts is the latency of a row of 32
// sources.  With a search per source, four loads in flight and a counter atomic
// per row of reverse pairs the largest of 1594 targets of 300k particles (10,000
// sources, Wendland C2) took 550 us of the loop; row_child, loads of eight rows
// (four with the velocities) and an atomic per four rows: 220 (the pool's 356 ->
// 203).  Keeping the sources in reach in shared memory costs another 85 us: most
// of these targets have more of them than fit.
template <int K>
__global__ void __launch_bounds__(kTWarps * 32) k_tree_density_fb(sphh::TreeDensityArgs a, PhysDev ph) {
  extern __shared__ __align__(16) unsigned char tsm[];
  const int warp = threadIdx.x >> 5, lane = threadIdx.x & 31;
  const NewtonConst& nwt = ph.newton;
  unsigned char* base = tsm + (size_t)warp * kTFbWarpSmem;
  float4* spos = reinterpret_cast<float4*>(base);
  uint32_t* sidx = reinterpret_cast<uint32_t*>(spos + kTCap);
  TPrune* pr = reinterpret_cast<TPrune*>(sidx + kTCap);
  const int32_t nq = min(*a.fb_count, (int32_t)a.n_total);
  unsigned long long pair_acc = 0;
  for (int32_t q = next_group(a.fb_work, lane); q < nq; q = next_group(a.fb_work, lane)) {
    const int32_t qe = a.fb_list[q];
    const bool own = (qe & kFbOwnLevel) != 0;
    const int32_t ti = qe & kFbIndex;
    const uint64_t key = a.skey[ti];
    const GridDev G = a.grid[sim_of_cell(a.grid, a.n_sims, (int32_t)(key >> 30))];
    const float4 reli = a.rel[ti];
    const int4 fi = a.fine[ti];
    const float4 vi = a.vel4[ti];
    if (qe & kFbPassive) {
      // outside the mask: the reverse pairs of its current support H to the
      // masked particles, from the finest level whose 27 cells hold it (the
      // top cells hold every support)
      const float hp = a.hs[ti];
      const float H = KernT<K>::gamma * hp;
      int dp = (int)a.level[ti];
      TreeLeaf Lp = cell_at_depth(key, dp);
      TGeo gp = leaf_geo(Lp, G);
      while (dp > 0 && hp > h_cap<K>(gp.side_d, gp.L)) {
        --dp;
        Lp = cell_at_depth(key, dp);
        gp = leaf_geo(Lp, G);
      }
      const float3 pp = rel_to(gp, reli, fi, kNoShift);
      const TRanges Rr = cell_ranges(G, Lp, a.skey, a.cell_start, lane);
      prune_tables(a.skey, Rr, Lp.depth, lane, pr);
      const float cs = Lp.depth < kTreeDepth ? 0.5f * gp.side : gp.side;
      const float H2 = H * H;
      const int2 hp2 = prune_round(lane, pp, H2 * (1.0f + 0x1p-10f), gp, cs, pr);
      const int nhp = hp2.x, tot = hp2.y;
      int ci = 0;
      for (int v0 = 0; v0 < tot; v0 += kTCap) {
        const int c = tstage_union(v0, tot, nhp, pr, lane, gp, a.rel, a.fine, spos, sidx, ci);
        for (int k0 = 0; k0 < c; k0 += 32) {
          const int k = k0 + lane;
          bool want = false;
          uint64_t rec = 0;
          if (k < c) {
            const float r2 = r2_of(pp, spos[k]);
            const uint32_t je = sidx[k];
            const int32_t j = unpack_j(je);
            want = a.act[j] != 0 && want_reverse(a, ti, j, r2, H2, H, gp.side);
            rec = reverse_rec(j, ti, unpack_s(je));
          }
          emit_warp(a, want, rec, lane);
        }
        __syncwarp();
      }
      continue;
    }
    // a target queued from its group starts at its own level from its
    // starting h; one that hit its level's cap one level coarser from the
    // capped h of the first solve
    float h = own ? a.hs[ti] : a.h[a.perm[ti]];
    bool conv = false, atcap = true;
    int passes = 0, d = (int)a.level[ti] - (own ? 0 : 1);
    if (d < 0) {
      // already at its top cell: the caller rebuilds the top grid from twice
      // the capped h; the first solve's other outputs stand
      if (lane == 0) {
        atomicOr(a.status, SPH_ST_REBUILD);
        a.fb_level[ti] = 0;
        a.h[a.perm[ti]] = 2.0f * h;
      }
      __syncwarp();
      continue;
    }
    TGeo g;
    TRanges R;
    float3 pi;
    bool one_chunk = true;
    int nh = 0, total = 0;
    float Rp = 0.0f, cside = 0.0f;
    // the sources: the children of the 27 cells whose box lies within the
    // selection radius Rp (with a margin far above the rounding of r); Rp =
    // min(cell side, 1.25 H) leaves room for the support to grow, and a support
    // beyond it selects again (H is warp-uniform).  Up to kTCap of them are
    // staged for the Newton passes, more are read again by each pass
    auto select = [&](float Hsup) {
      if (!(Hsup > Rp)) return;
      Rp = fminf(g.side, 1.25f * Hsup);
      const int2 hit = prune_round(lane, pi, Rp * Rp * (1.0f + 0x1p-10f), g, cside, pr);
      nh = hit.x;
      total = hit.y;
      one_chunk = total <= kTCap;
      int ci = 0;
      if (one_chunk) tstage_union(0, total, nh, pr, lane, g, a.rel, a.fine, spos, sidx, ci);
    };
    for (; d >= 0; --d) {
      const TreeLeaf Lc = cell_at_depth(key, d);
      g = leaf_geo(Lc, G);
      R = cell_ranges(G, Lc, a.skey, a.cell_start, lane);
      pi = rel_to(g, reli, fi, kNoShift);
      const float hcap = h_cap<K>(g.side_d, g.L);
      prune_tables(a.skey, R, Lc.depth, lane, pr);
      cside = Lc.depth < kTreeDepth ? 0.5f * g.side : g.side;
      Rp = 0.0f;  // nothing selected at this level yet
      float hlo = 0.0f, hhi = INFINITY;
      int it = 0;
      if (h > hcap) h = hcap;
      bool done = false;
      while (!done) {  // warp-uniform: every lane holds the same reduced sums
        const float H = KernT<K>::gamma * h;
        select(H);
        const float Hinv = 1.0f / H;
        float Sw = 0.f, Sdw = 0.f;
        if (one_chunk) {
          for (int k = lane; k < total; k += 32) tnewton_pair<K>(r2_of(pi, spos[k]), H, Hinv, Sw, Sdw);
        } else {
          const float2 S = tnewton_stream<K>(total, nh, pr, lane, g, pi, H, Hinv, a.rel, a.fine);
          Sw = S.x;
          Sdw = S.y;
        }
        Sw = wsum(Sw);
        Sdw = wsum(Sdw);
        ++passes;
        done = newton_update(Sw, Sdw, nwt, hcap, h, hlo, hhi, it, atcap, conv);
      }
      if (!atcap) break;
    }
    if (d < 0) {
      // even the top cell is too small: the caller rebuilds the top grid
      if (lane == 0) atomicOr(a.status, SPH_ST_REBUILD);
      d = 0;
    }
    // final pass at h, reverse pairs of this target
    const float H = KernT<K>::gamma * h;
    select(H);
    const float Hinv = 1.0f / H;
    const float H2 = H * H;
    TDSums s;
    tds_zero(s);
    int ci = 0;
#pragma unroll 1
    for (int u0 = 0; u0 < total; u0 += 4 * 32) {
      float4 rj[4], vj[4];
      int4 fj[4], sj[4];
      uint32_t je[4];
#pragma unroll
      for (int i = 0; i < 4; ++i) {
        const int c = row_child(u0 + 32 * i, nh, pr, lane, ci);
        sj[i] = pr->src[c];
        const int32_t j = sj[i].x + min(u0 + 32 * i + lane, total - 1);
        je[i] = pack_js(j, child_shift(pr, c));
        rj[i] = a.rel[j];
        fj[i] = a.fine[j];
        vj[i] = a.vel4[j];
      }
      unsigned want = 0;
#pragma unroll
      for (int i = 0; i < 4; ++i) {
        const float3 pj = item_pos(g, rj[i], fj[i], sj[i]);
        const float dx = pi.x - pj.x, dy = pi.y - pj.y, dz = pi.z - pj.z;
        const float r2 = fmaf(dx, dx, fmaf(dy, dy, dz * dz));
        if (u0 + 32 * i + lane < total && r2 < H2) {
          tdens_pair<K>(dx, dy, dz, vi, vj[i], rj[i].w, H, Hinv, s);
          if (want_reverse_t(__int_as_float(fj[i].w), ti, unpack_j(je[i]), r2, H2, H, g.side)) want |= 1u << i;
        }
      }
      emit_rows(a, want, je, ti, lane);
    }
    s.w = wsum(s.w);
    s.dw = wsum(s.dw);
    s.mw = wsum(s.mw);
    s.mdw = wsum(s.mdw);
    s.div = wsum(s.div);
    s.cx = wsum(s.cx);
    s.cy = wsum(s.cy);
    s.cz = wsum(s.cz);
    s.npair = wsumi(s.npair);
    if (lane == 0) {
      tdens_write<K>(a, ph, ti, h, s, vi.w, passes, !conv && !atcap);
      if (atcap) a.h[a.perm[ti]] = 2.0f * h;  // next starting guess
      a.fb_level[ti] = (int8_t)d;
      pair_acc += (unsigned long long)s.npair;
    }
    __syncwarp();
  }
  if (ph.count_pairs && lane == 0 && pair_acc) atomicAdd(a.pairs, pair_acc);
}

// The force on the targets of k_tree_density_fb, a warp each, and as there bound
// by the latency of the largest.  The reach's sources are tested 128 at a time,
// and those in reach gathered into full warps of pairs.  Against a walk child by
// child with the ranges searched one after another: 229 -> 145 us in the pool of
// 48 boxes, 189 -> 109 us for 300k particles with Wendland C2.  A CTA per target
// (the set-up by one warp) took 183 and 105.
template <int kFl, int K>
__global__ void __launch_bounds__(kTWarps * 32) k_tree_force_fb(sphh::TreeForceArgs a, PhysDev ph, SphenixDev x) {
  __shared__ TPrune prune[kTWarps];
  __shared__ uint32_t rings[kTWarps][64];
  const int lane = threadIdx.x & 31;
  TPrune* pr = &prune[threadIdx.x >> 5];
  uint32_t* ring = rings[threadIdx.x >> 5];
  const int32_t nq = min(*a.fb_count, (int32_t)a.n_total);
  unsigned long long pair_acc = 0;
  for (int32_t q = next_group(a.fb_work, lane); q < nq; q = next_group(a.fb_work, lane)) {
    const int32_t qe = a.fb_list[q];
    if (qe & kFbPassive) continue;  // outside the mask: no force
    const int32_t ti = qe & kFbIndex;
    const uint64_t key = a.skey[ti];
    const int sim = sim_of_cell(a.grid, a.n_sims, (int32_t)(key >> 30));
    const GridDev G = a.grid[sim];
    const TreeLeaf Lc = cell_at_depth(key, (int)a.fb_level[ti]);
    const TGeo g = leaf_geo(Lc, G);
    const float dt = kFl == kTGradient ? (float)(x.dt_dev != nullptr ? x.dt_dev[sim] : x.dt) : 0.0f;
    const TRec hi = trec_head(a, ti);
    const float3 pi = rec_rel_to(g, hi, kNoShift);
    const float4 vi = trec_vel(a, ti);
    const float4 ci = trec_pres(a, ti);
    const float4 ei = kFl != kTMin ? a.fE[ti] : make_float4(0.f, 0.f, 0.f, 0.f);
    const float2 di = make_float2(__int_as_float(hi.q1.w), __frcp_rn(hi.q0.w));
    const float Hi = hi.q0.w;
    // own reach: the list radius, or the support where it outgrew the list
    // (both within the cell of the fallback level, whose 27 cells hold every
    // source closer than that); the sources beyond it with a larger support
    // sent their pairs as reverse pairs (each emitted from r >= the list radius)
    const float C = fmaxf(a.lrad[ti], Hi);
    const float C2 = C * C;
    TFSums s;
    s.ax = s.ay = s.az = s.du = s.vsig = 0.f;
    s.npair = 0;
    if (kFl == kTGradient) s.ay = ei.y;
    // the pairs in reach wait in a ring until there is one for every lane
    int head = 0, np = 0;
    auto walk = [&](int cnt) {
      if (lane < cnt) {
        const uint32_t je = ring[(head + lane) & 63];
        const int32_t j = unpack_j(je);
        const TRec hj = trec_head(a, j);
        const float3 pj = rec_rel_to(g, hj, unpack_s(je));
        tforce_rec<kFl, K>(pi.x - pj.x, pi.y - pj.y, pi.z - pj.z, vi, ci, ei, Hi, di.y, di.x, a, j, hj, ph, s);
      }
    };
    auto push = [&](bool in, uint32_t je) {
      const unsigned m = __ballot_sync(0xffffffffu, in);
      if (in) ring[(head + np + __popc(m & ((1u << lane) - 1u))) & 63] = je;
      np += __popc(m);
      __syncwarp();
      if (np >= 32) {
        walk(32);
        head += 32;
        np -= 32;
        __syncwarp();
      }
    };
    const float cside = Lc.depth < kTreeDepth ? 0.5f * g.side : g.side;
    const TRanges R = cell_ranges(G, Lc, a.skey, a.cell_start, lane);
    prune_tables(a.skey, R, Lc.depth, lane, pr);
    // (a margin far above the rounding of r)
    const int2 hit = prune_round(lane, pi, C2 * (1.0f + 0x1p-10f), g, cside, pr);
    int at = 0;
#pragma unroll 1
    for (int u0 = 0; u0 < hit.y; u0 += 4 * 32) {
      uint32_t je[4];
      bool in[4];
      int4 sj[4];
      TRec hj[4];
#pragma unroll
      for (int i = 0; i < 4; ++i) {
        const int c = row_child(u0 + 32 * i, hit.x, pr, lane, at);
        sj[i] = pr->src[c];
        const int32_t j = sj[i].x + min(u0 + 32 * i + lane, hit.y - 1);
        je[i] = pack_js(j, child_shift(pr, c));
        hj[i] = trec_head(a, j);
      }
#pragma unroll
      for (int i = 0; i < 4; ++i) {
        const float3 pj = item_pos(g, hj[i].q0, hj[i].q1, sj[i]);
        const float dx = pi.x - pj.x, dy = pi.y - pj.y, dz = pi.z - pj.z;
        in[i] = u0 + 32 * i + lane < hit.y && unpack_j(je[i]) != ti && fmaf(dx, dx, fmaf(dy, dy, dz * dz)) < C2;
      }
#pragma unroll 1
      for (int i = 0; i < 4; ++i) push(i == 0 ? in[0] : i == 1 ? in[1] : i == 2 ? in[2] : in[3],
                                       i == 0 ? je[0] : i == 1 ? je[1] : i == 2 ? je[2] : je[3]);
    }
    if (kFl != kTGradient) {
      const int32_t r0 = a.rev_start[ti], r1 = a.rev_start[ti + 1];
#pragma unroll 1
      for (int32_t k0 = r0; k0 < r1; k0 += 32) {
        bool in = false;
        uint32_t je = 0;
        if (k0 + lane < r1) {
          je = a.rev[k0 + lane];
          const float3 pj = rec_rel_to(g, trec_head(a, unpack_j(je)), unpack_s(je));
          const float dx = pi.x - pj.x, dy = pi.y - pj.y, dz = pi.z - pj.z;
          in = fmaf(dx, dx, fmaf(dy, dy, dz * dz)) >= C2;
        }
        push(in, je);
      }
    }
    walk(np);
    __syncwarp();
    s.ax = wsum(s.ax);
    if (kFl == kTGradient) {
#pragma unroll
      for (int o = 16; o > 0; o >>= 1) s.ay = fmaxf(s.ay, __shfl_xor_sync(0xffffffffu, s.ay, o));
    } else {
      s.ay = wsum(s.ay);
    }
    s.az = wsum(s.az);
    s.du = wsum(s.du);
#pragma unroll
    for (int o = 16; o > 0; o >>= 1) s.vsig = fmaxf(s.vsig, __shfl_xor_sync(0xffffffffu, s.vsig, o));
    s.npair = wsumi(s.npair);
    if (lane == 0) {
      tforce_write<kFl>(a, x, dt, ti, Hi, ei, s);
      pair_acc += (unsigned long long)s.npair;
    }
  }
  if (ph.count_pairs && a.pairs != nullptr && lane == 0 && pair_acc) atomicAdd(a.pairs, pair_acc);
}

}  // namespace sphk

namespace sphh {
using namespace sphk;

__global__ void k_tree_mask(int64_t n, const int32_t* __restrict__ perm, const uint8_t* __restrict__ active,
                            uint8_t* __restrict__ out) {
  for (int64_t k = (int64_t)blockIdx.x * blockDim.x + threadIdx.x; k < n; k += (int64_t)gridDim.x * blockDim.x)
    out[k] = active[perm[k]] != 0 ? 1 : 0;
}

static int tree_blocks(int64_t n) {
  int64_t b = (n + 255) / 256;
  return (int)(b < 1 ? 1 : (b > 65535 ? 65535 : b));
}

cudaError_t sort_reverse_pairs(int64_t n, const int32_t* start, uint32_t* rev, int32_t* queue, int32_t* n_mid,
                               int32_t* n_long, int num_sms, cudaStream_t st) {
  cudaError_t e = cudaMemsetAsync(n_mid, 0, sizeof(int32_t), st);
  if (e == cudaSuccess) e = cudaMemsetAsync(n_long, 0, sizeof(int32_t), st);
  if (e != cudaSuccess) return e;
  k_rev_sort<<<tree_blocks(n), kRevThreads, 0, st>>>(n, start, rev, queue, n_mid, n_long);
  k_rev_mid<<<num_sms * 6, kRevThreads, 0, st>>>(start, rev, queue, n_mid);
  k_rev_long<<<num_sms * 4, kRevThreads, 0, st>>>(n, start, rev, queue, n_long);
  return cudaGetLastError();
}

template <int K>
static cudaError_t launch_tree_density_k(const TreeDensityArgs& a, const PhysDev& ph, cudaStream_t st) {
  static PerDevice<2> known;
  int bps[2];  // resident blocks of the main and of the per-target kernel
  cudaError_t e = known.get(bps, [](int (&v)[2]) {
    cudaError_t r = opt_in(k_tree_density<K, false>, kTDensSmem);
    if (r == cudaSuccess) r = opt_in(k_tree_density<K, true>, kTDensSmem);
    if (r == cudaSuccess) r = opt_in(k_tree_density_fb<K>, kTFbSmem);
    if (r == cudaSuccess) r = resident_blocks(k_tree_density<K, false>, kTWarps * 32, kTDensSmem, &v[0]);
    if (r == cudaSuccess) r = resident_blocks(k_tree_density_fb<K>, kTWarps * 32, kTFbSmem, &v[1]);
    return r;
  });
  const int64_t n = a.n_total;
  if (e == cudaSuccess) e = cudaMemsetAsync(a.rev_count, 0, sizeof(unsigned long long), st);
  if (e == cudaSuccess) e = cudaMemsetAsync(a.work, 0, sizeof(int32_t), st);
  if (e == cudaSuccess) e = cudaMemsetAsync(a.fb_count, 0, sizeof(int32_t), st);
  if (e == cudaSuccess) e = cudaMemsetAsync(a.fb_work, 0, sizeof(int32_t), st);
  if (e == cudaSuccess) e = cudaMemsetAsync(a.rev_fill, 0, sizeof(int32_t) * (n > 0 ? n : 1), st);
  if (e != cudaSuccess) return e;
  if (n <= 0) return cudaSuccess;
  const int64_t want = (n + (int64_t)kTWin * kTWarps - 1) / ((int64_t)kTWin * kTWarps);
  const int blocks = (int)(want < (int64_t)a.num_sms * bps[0] ? want : (int64_t)a.num_sms * bps[0]);
  if (a.act != nullptr)
    k_tree_density<K, true><<<blocks, kTWarps * 32, kTDensSmem, st>>>(a, ph);
  else
    k_tree_density<K, false><<<blocks, kTWarps * 32, kTDensSmem, st>>>(a, ph);
  k_tree_density_fb<K><<<a.num_sms * bps[1], kTWarps * 32, kTFbSmem, st>>>(a, ph);
  e = scan_exclusive(a.rev_fill, a.rev_start, n, a.scan_tmp, a.num_sms, st);
  if (e == cudaSuccess) e = cudaMemsetAsync(a.rev_fill, 0, sizeof(int32_t) * n, st);
  if (e != cudaSuccess) return e;
  k_rev_scatter<<<a.num_sms * 4, 256, 0, st>>>(a.rev_raw, a.rev_count, a.rev_cap, a.rev_start, a.rev_fill, a.rev);
  // (the scatter's cursors and the work counters are free again)
  return sort_reverse_pairs(n, a.rev_start, a.rev, a.rev_fill, a.work, a.fb_work, a.num_sms, st);
}

template <int kFl, int K>
static cudaError_t launch_tree_force_k(const TreeForceArgs& a, const PhysDev& ph, const SphenixDev& x,
                                       cudaStream_t st) {
  static PerDevice<1> known;
  int bps[1];
  cudaError_t e =
      known.get(bps, [](int (&v)[1]) { return resident_blocks(k_tree_force<kFl, K>, kTWarps * 32, 0, &v[0]); });
  if (e == cudaSuccess) e = cudaMemsetAsync(a.work, 0, sizeof(int32_t), st);
  if (e == cudaSuccess) e = cudaMemsetAsync(a.fb_work, 0, sizeof(int32_t), st);
  if (e != cudaSuccess) return e;
  // windows of two rounds; of one while that does not fill the resident warps
  // four times (6,000 particles 317 -> 302 us; 1M masked 1.59 -> 1.66 ms)
  const int64_t warps = (int64_t)a.num_sms * bps[0] * kTWarps;
  int win = a.n_total < warps * 4 * kTPer ? kTPer : 2 * kTPer;
  // masked loops skip most rounds, and then the windows' counter is what costs: of
  // four rounds where that leaves each warp eight windows (1M particles, 0.1 % of
  // them masked: 182 -> 139 us, a leaf per warp 156; all of them: 735 and 732; 300k,
  // two windows a warp, half of them masked: 251 -> 259)
  if (a.act != nullptr && a.n_total >= warps * 8 * 4 * kTPer) win = 4 * kTPer;
  const int64_t want = (a.n_total + (int64_t)win * kTWarps - 1) / ((int64_t)win * kTWarps);
  const int blocks = (int)(want < (int64_t)a.num_sms * bps[0] ? want : (int64_t)a.num_sms * bps[0]);
  k_tree_force<kFl, K><<<blocks < 1 ? 1 : blocks, kTWarps * 32, 0, st>>>(a, ph, x, win);
  k_tree_force_fb<kFl, K><<<a.num_sms * bps[0], kTWarps * 32, 0, st>>>(a, ph, x);
  return cudaGetLastError();
}

template <int kFl>
static cudaError_t launch_tree_force_fl(const TreeForceArgs& a, const PhysDev& ph, const SphenixDev& x,
                                        cudaStream_t st) {
  switch (ph.kernel) {
    case kKernQuartic:
      return launch_tree_force_k<kFl, kKernQuartic>(a, ph, x, st);
    case kKernWendlandC2:
      return launch_tree_force_k<kFl, kKernWendlandC2>(a, ph, x, st);
    default:
      return launch_tree_force_k<kFl, kKernCubic>(a, ph, x, st);
  }
}

cudaError_t launch_tree_sphenix_force(const TreeForceArgs& a, const PhysDev& ph, const SphenixDev& x,
                                      cudaStream_t st) {
  if (a.fE == nullptr) return cudaErrorInvalidValue;
  return launch_tree_force_fl<kTSphenix>(a, ph, x, st);
}

cudaError_t launch_tree_sphenix_gradient(const TreeForceArgs& a, const PhysDev& ph, const SphenixDev& x,
                                         cudaStream_t st) {
  if (a.fE == nullptr || a.alpha_c_out == nullptr) return cudaErrorInvalidValue;
  return launch_tree_force_fl<kTGradient>(a, ph, x, st);
}

cudaError_t launch_tree_density(const TreeDensityArgs& a, const PhysDev& ph, cudaStream_t st) {
  switch (ph.kernel) {
    case kKernQuartic:
      return launch_tree_density_k<kKernQuartic>(a, ph, st);
    case kKernWendlandC2:
      return launch_tree_density_k<kKernWendlandC2>(a, ph, st);
    default:
      return launch_tree_density_k<kKernCubic>(a, ph, st);
  }
}

cudaError_t launch_tree_force(const TreeForceArgs& a, const PhysDev& ph, cudaStream_t st) {
  return launch_tree_force_fl<kTMin>(a, ph, SphenixDev{}, st);
}

cudaError_t launch_tree_limit(const TreeForceArgs& a, const PhysDev& ph, cudaStream_t st) {
  if (a.fE == nullptr || a.bins_out == nullptr) return cudaErrorInvalidValue;
  return launch_tree_force_fl<kTLimit>(a, ph, SphenixDev{}, st);
}

cudaError_t launch_tree_wake(const TreeForceArgs& a, const PhysDev& ph, cudaStream_t st) {
  if (a.fE == nullptr || a.act == nullptr || a.wake == nullptr) return cudaErrorInvalidValue;
  return launch_tree_force_fl<kTWake>(a, ph, SphenixDev{}, st);
}

cudaError_t launch_tree_mask(int64_t n, const int32_t* perm, const uint8_t* active, uint8_t* out, int32_t* pre,
                             int32_t* tmp, int num_sms, cudaStream_t st) {
  if (n <= 0) return cudaSuccess;
  k_tree_mask<<<tree_blocks(n), 256, 0, st>>>(n, perm, active, out);
  if (pre != nullptr) {
    const cudaError_t e = scan_exclusive(out, pre, n, tmp, num_sms, st);
    if (e != cudaSuccess) return e;
  }
  return cudaGetLastError();
}

}  // namespace sphh
