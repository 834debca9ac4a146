// fof.cu -- friends-of-friends groups (Sec. 7.1) on the uniform cell grid.
//
// Particles i and j are friends when their minimum-image distance is below
// the linking length b; groups are the connected components (union-find,
// Sec. 7.1).  The grid's cells are at least b wide, so friends lie in the
// same or adjacent cells; every pair is visited once: from the particle of
// the lower sorted slot inside a cell, and across the 13 axes delta_q (the
// other 13 neighbours see the pair from the opposite side).
//
// The decision is the FP64 one of the definition (d = x_i - x_j wrapped once
// into [-L/2, L/2], r2 = dx*dx + dy*dy + dz*dz, r2 < b*b, no contraction).
// An FP32 distance from cell-relative positions settles every pair whose r2
// is farther from b^2 than its rounding can reach; the rest take the FP64
// test, so the links are exactly those of the definition.
//
// Dense cells.  Particles of one octant of a cell are friends as they are: an
// octant's diagonal is 0.866 cells, below b while cells are at most 1.15 b wide.
// A cell of at least kFofDense particles has its particles ordered by octant and
// each octant's particles start as one set; two octants (or an octant and a
// particle) are then linked by their first friendly pair, if they are not one
// set yet.  A core of thousands of particles within b of each other so takes a
// few root checks per octant instead of a union per pair, all of them contending
// for the same root (the 1M clustered box: 7.5 ms for all pairs, 0.73 ms for the
// octants and the rest; the call 8.2 -> 1.15 ms, cell_start and the sort included).
//
// Union-find on the caller's group array, lock-free: a set's root is its
// smallest index, a union hooks the larger root below the smaller one with
// one compare-and-swap (retried when the root changed meanwhile), and the
// link pass's finds halve their paths.  Every parent pointer only ever moves to an
// ancestor, so concurrent halving and hooking keep a valid forest, and the final
// roots are the groups' smallest indices whatever the order of the unions.  The
// parent loads bypass L1 (other SMs write them).  Loops are bounded; a
// bound that is hit sets SPH_ST_CAPACITY.
#include "sph_internal.cuh"
#include "sph_launch.h"

namespace sphk {

constexpr int kFofMaxSteps = 1 << 20;  // bound of one find or one union's retries

// kHalve: path halving (the link pass).  The label pass reads only: there
// every particle's entry is overwritten with its root while other threads
// walk through it, and a halving write arriving after that would replace a
// final root by a mere ancestor.
template <bool kHalve>
__device__ __forceinline__ int32_t fof_find(int32_t* parent, int32_t x, int32_t* status) {
  for (int it = 0; it < kFofMaxSteps; ++it) {
    const int32_t p = __ldcg(parent + x);
    if (p == x) return x;
    const int32_t gp = __ldcg(parent + p);
    if (kHalve && gp != p) __stcg(parent + x, gp);  // gp is an ancestor of x
    x = gp;
  }
  atomicOr(status, SPH_ST_CAPACITY);
  return x;
}

// Joins the sets of a and b; returns a root that both had at some time since.
__device__ __noinline__ int32_t fof_union(int32_t* parent, int32_t a, int32_t b, int32_t* status) {
  for (int it = 0; it < kFofMaxSteps; ++it) {
    a = fof_find<true>(parent, a, status);
    b = fof_find<true>(parent, b, status);
    if (a == b) return a;
    if (a > b) {
      const int32_t t = a;
      a = b;
      b = t;
    }
    if (atomicCAS(parent + b, b, a) == b) return a;  // b was still a root: hooked
  }
  atomicOr(status, SPH_ST_CAPACITY);
  return a;
}

// Whether b is known to be in the set of ancestor `root` of another particle: one
// load where two finds take four.
__device__ __forceinline__ bool fof_joined(const int32_t* parent, int32_t root, int32_t b) {
  return __ldcg(parent + b) == root;
}

// FP64 friendship test of the definition (minimum image, no contraction).
__device__ __forceinline__ double fof_min_image(double d, double L) {
  if (d > 0.5 * L) return __dadd_rn(d, -L);
  if (d < -0.5 * L) return __dadd_rn(d, L);
  return d;
}

__device__ __forceinline__ bool fof_friends64(const double* x, const double* y, const double* z, int32_t i,
                                              int32_t j, double L, double b2) {
  const double dx = fof_min_image(__dadd_rn(x[i], -x[j]), L);
  const double dy = fof_min_image(__dadd_rn(y[i], -y[j]), L);
  const double dz = fof_min_image(__dadd_rn(z[i], -z[j]), L);
  const double r2 = __dadd_rn(__dadd_rn(__dmul_rn(dx, dx), __dmul_rn(dy, dy)), __dmul_rn(dz, dz));
  return r2 < b2;
}

constexpr int kFofDense = 16;  // particles of a cell taken by octants

// Whether octants are sets as they are (with a margin far above the rounding of
// the FP32 positions that decide the octant).
__device__ __forceinline__ bool fof_octants(const GridDev& G, double b) { return 0.86603 * 1.0001 * G.cell < b; }

// Sorted cell-relative positions (index in .w) and singleton sets; the cells
// taken by octants are queued, their positions to `rel0` to be ordered.
__global__ void k_fof_prep(sphh::FofArgs a) {
  const GridDev G = a.grid[0];
  const bool oct = fof_octants(G, a.link);
  for (int64_t s = (int64_t)blockIdx.x * blockDim.x + threadIdx.x; s < a.n_total;
       s += (int64_t)gridDim.x * blockDim.x) {
    const int32_t p = a.perm[s];
    const int32_t cg = a.key[p], c = cg - G.cell_base;
    const int32_t kx = c % G.n_c, ky = (c / G.n_c) % G.n_c, kz = c / (G.n_c * G.n_c);
    const float4 r = make_float4((float)(a.x[p] - (double)kx * G.cell), (float)(a.y[p] - (double)ky * G.cell),
                                 (float)(a.z[p] - (double)kz * G.cell), __int_as_float(p));
    const int32_t t0 = a.cell_start[cg];
    const bool dense = oct && a.cell_start[cg + 1] - t0 >= kFofDense;
    (dense ? a.rel0 : a.rel)[s] = r;
    if (dense) {
      if (s == t0) a.queue[atomicAdd(a.queued, 1)] = cg;
    } else {
      a.group[p] = p;
    }
  }
}

__device__ __forceinline__ int fof_octant(const float4& r, float half) {
  return (r.x >= half ? 1 : 0) | (r.y >= half ? 2 : 0) | (r.z >= half ? 4 : 0);
}

// A queued cell's particles in order of octant, then index (a warp per cell);
// an octant's particles hang from its first, the smallest index.  The octants'
// first places go to oct[first place of the cell + octant].
__global__ void k_fof_octants(sphh::FofArgs a) {
  const GridDev G = a.grid[0];
  const int lane = threadIdx.x & 31;
  const unsigned lt = (1u << lane) - 1u;
  const float half = 0.5f * G.cell_f;
  const int32_t nq = *a.queued;
  for (int32_t q = (blockIdx.x * blockDim.x + threadIdx.x) >> 5; q < nq; q += (gridDim.x * blockDim.x) >> 5) {
    const int32_t cg = a.queue[q], t0 = a.cell_start[cg], t1 = a.cell_start[cg + 1];
    int32_t mine = 0;  // lane o < 8: particles of octant o
    for (int32_t t = t0; t < t1; t += 32) {
      const int o = t + lane < t1 ? fof_octant(a.rel0[t + lane], half) : 8;
#pragma unroll
      for (int k = 0; k < 8; ++k) {
        const int m = __popc(__ballot_sync(0xffffffffu, o == k));
        if (lane == k) mine += m;
      }
    }
    int32_t at = mine;  // exclusive prefix: the octants' first places
#pragma unroll
    for (int o = 1; o < 8; o <<= 1) {
      const int32_t v = __shfl_up_sync(0xffffffffu, at, o);
      if (lane >= o) at += v;
    }
    at += t0 - mine;
    if (lane < 8) a.oct[t0 + lane] = at;
    int32_t root = 0;  // lane o < 8: octant o's first index
    bool any = false;
    for (int32_t t = t0; t < t1; t += 32) {
      const bool ok = t + lane < t1;
      const float4 r = ok ? a.rel0[t + lane] : make_float4(0.f, 0.f, 0.f, 0.f);
      const int o = ok ? fof_octant(r, half) : 8;
      const int32_t p = __float_as_int(r.w);
      int32_t to = 0, top = 0;
#pragma unroll
      for (int k = 0; k < 8; ++k) {
        const unsigned m = __ballot_sync(0xffffffffu, o == k);
        const int32_t first = __shfl_sync(0xffffffffu, p, m != 0u ? __ffs((int)m) - 1 : 0);
        if (lane == k && m != 0u && !any) {
          any = true;
          root = first;
        }
        const int32_t base = __shfl_sync(0xffffffffu, at, k), r0 = __shfl_sync(0xffffffffu, root, k);
        if (o == k) {
          to = base + __popc(m & lt);
          top = r0;
        }
        if (lane == k) at += __popc(m);
      }
      if (ok) {
        a.rel[to] = r;
        a.group[p] = top;
      }
    }
  }
}

// Neighbour cell o of cell (kx, ky, kz): itself (0) or along the 13 axes; its
// range of sorted places and its offset in cells.
struct FofCell {
  int32_t t0, t1;
  float ox, oy, oz;
};
__device__ __forceinline__ FofCell fof_cell(const sphh::FofArgs& a, const GridDev& G, int32_t kx, int32_t ky,
                                            int32_t kz, int o) {
  const int32_t nc = G.n_c;
  int dx = 0, dy = 0, dz = 0;
  if (o > 0) axis_delta(o - 1, dx, dy, dz);
  int32_t cx = kx + dx, cy = ky + dy, cz = kz + dz;
  cx += cx < 0 ? nc : 0;
  cx -= cx >= nc ? nc : 0;
  cy += cy < 0 ? nc : 0;
  cy -= cy >= nc ? nc : 0;
  cz += cz < 0 ? nc : 0;
  cz -= cz >= nc ? nc : 0;
  const int32_t cn = G.cell_base + cx + nc * (cy + nc * cz);
  return {a.cell_start[cn], a.cell_start[cn + 1], (float)dx * G.cell_f, (float)dy * G.cell_f, (float)dz * G.cell_f};
}

// FP32 distances of cell-relative coordinates (|x| below two cells) are within
// ~1e-6 (2 cell)^2 of the true r2: a band of that width around b^2, plus a
// margin, goes to the FP64 test.
struct FofTest {
  float lo, hi;
  double b2;
};
__device__ __forceinline__ FofTest fof_test(const GridDev& G, double link) {
  const double b2 = link * link;
  const float band = 4e-6f * (2.0f * G.cell_f) * (2.0f * G.cell_f) + 1e-5f * (float)b2;
  return {(float)b2 - band, (float)b2 + band, b2};
}
__device__ __forceinline__ bool fof_friends(const sphh::FofArgs& a, const GridDev& G, const FofTest& T, const float4& p,
                                            const float4& q, const FofCell& C) {
  const float fx = p.x - (q.x + C.ox), fy = p.y - (q.y + C.oy), fz = p.z - (q.z + C.oz);
  const float r2 = fmaf(fx, fx, fmaf(fy, fy, fz * fz));
  if (r2 >= T.hi) return false;
  return r2 < T.lo || fof_friends64(a.x, a.y, a.z, __float_as_int(p.w), __float_as_int(q.w), G.L, T.b2);
}

// Gap along one axis between [p0, p1] and octant bit `bit` of a cell at offset
// off (both in cell-relative units).
__device__ __forceinline__ float fof_gap(float p0, float p1, float off, int bit, float half) {
  const float lo = off + (bit ? half : 0.0f);
  return fmaxf(fmaxf(lo - p1, p0 - (lo + half)), 0.0f);
}

// Particles of cells not taken by octants, a thread each: the later particles
// of the cell and those of the 13 neighbours (or their octants, which the warp
// searches together).  Bound by latency: the empty rows skipped, four particles'
// loads in flight, one load instead of two finds for a pair that is joined
// already, and twelve blocks of 128 threads per SM took the 1M clustered box from
// 508 to 388 us.
__global__ void __launch_bounds__(128, 12) k_fof_link(sphh::FofArgs a) {
  const GridDev G = a.grid[0];
  const int32_t nc = G.n_c;
  const FofTest T = fof_test(G, a.link);
  const int dense = fof_octants(G, a.link) ? kFofDense : INT32_MAX;
  const float half = 0.5f * G.cell_f;
  const int lane = threadIdx.x & 31;
  for (int64_t w = (int64_t)blockIdx.x * blockDim.x + threadIdx.x - lane; w < a.n_total;
       w += (int64_t)gridDim.x * blockDim.x) {
    const int64_t s = w + lane;
    bool on = s < a.n_total;
    const int32_t pi = on ? a.perm[s] : 0;
    const int32_t cg = on ? a.key[pi] : G.cell_base, c = cg - G.cell_base;
    on = on && a.cell_start[cg + 1] - a.cell_start[cg] < dense;
    const float4 me = on ? a.rel[s] : make_float4(0.f, 0.f, 0.f, 0.f);
    const int32_t kx = c % nc, ky = (c / nc) % nc, kz = c / (nc * nc);
    int32_t root = on ? fof_find<true>(a.group, pi, a.status) : 0;  // an ancestor of pi
    // the neighbours beyond the own row lie in four rows of three cells, one
    // after another in memory: a row without particles is skipped (most are, of
    // cells of the linking length), and all rows' ends are in flight together
    unsigned todo = on ? (1u << (kAxes + 1)) - 1u : 0u;
    if (on && kx > 0 && kx < nc - 1) {
      int32_t r0[4], r1[4];
#pragma unroll
      for (int k = 0; k < 4; ++k) {
        const int dy = k == 0 ? 1 : k - 2, dz = k == 0 ? 0 : 1;
        int32_t cy = ky + dy, cz = kz + dz;
        cy += cy < 0 ? nc : 0;
        cy -= cy >= nc ? nc : 0;
        cz -= cz >= nc ? nc : 0;
        const int32_t cn = G.cell_base + kx - 1 + nc * (cy + nc * cz);
        r0[k] = a.cell_start[cn];
        r1[k] = a.cell_start[cn + 3];
      }
#pragma unroll
      for (int k = 0; k < 4; ++k)
        if (r0[k] == r1[k]) todo &= ~(7u << (2 + 3 * k));
    }
    for (unsigned all = __reduce_or_sync(0xffffffffu, todo); all != 0u; all &= all - 1u) {
      const int o = __ffs((int)all) - 1;
      FofCell C = {0, 0, 0.f, 0.f, 0.f};
      if ((todo >> o) & 1u) C = fof_cell(a, G, kx, ky, kz, o);
      const bool octs = C.t1 - C.t0 >= dense;
      if (!octs) {
        if (o == 0) C.t0 = (int32_t)s + 1;
        for (int32_t t = C.t0; t < C.t1; t += 4) {
          int32_t pq[4], up[4];
#pragma unroll
          for (int i = 0; i < 4; ++i) {
            const float4 q = a.rel[min(t + i, C.t1 - 1)];
            pq[i] = t + i < C.t1 && fof_friends(a, G, T, me, q, C) ? __float_as_int(q.w) : -1;
          }
#pragma unroll
          for (int i = 0; i < 4; ++i) up[i] = pq[i] >= 0 ? __ldcg(a.group + pq[i]) : 0;
#pragma unroll
          for (int i = 0; i < 4; ++i)
            if (pq[i] >= 0 && up[i] != root) root = fof_union(a.group, pi, pq[i], a.status);
        }
      }
      if (!__any_sync(0xffffffffu, octs)) continue;
      // octants within reach that are not in this particle's set yet, searched
      // for a friend by the whole warp
#pragma unroll 1
      for (int k = 0; k < 8; ++k) {
        int32_t u0 = 0, u1 = 0, pk = 0;
        bool open = octs;
        if (open) {
          u0 = a.oct[C.t0 + k];
          u1 = k < 7 ? a.oct[C.t0 + k + 1] : C.t1;
          const float gx = fof_gap(me.x, me.x, C.ox, k & 1, half), gy = fof_gap(me.y, me.y, C.oy, (k >> 1) & 1, half),
                      gz = fof_gap(me.z, me.z, C.oz, k >> 2, half);
          open = u0 < u1 && fmaf(gx, gx, fmaf(gy, gy, gz * gz)) < T.hi;
        }
        if (open) {
          pk = __float_as_int(a.rel[u0].w);
          open = !fof_joined(a.group, root, pk) &&
                 fof_find<true>(a.group, pi, a.status) != fof_find<true>(a.group, pk, a.status);
        }
        for (unsigned left = __ballot_sync(0xffffffffu, open); left != 0u; left &= left - 1u) {
          const int l = __ffs((int)left) - 1;
          const float4 p = make_float4(__shfl_sync(0xffffffffu, me.x, l), __shfl_sync(0xffffffffu, me.y, l),
                                       __shfl_sync(0xffffffffu, me.z, l), __shfl_sync(0xffffffffu, me.w, l));
          const int32_t v0 = __shfl_sync(0xffffffffu, u0, l), v1 = __shfl_sync(0xffffffffu, u1, l);
          const FofCell D = {v0, v1, __shfl_sync(0xffffffffu, C.ox, l), __shfl_sync(0xffffffffu, C.oy, l),
                             __shfl_sync(0xffffffffu, C.oz, l)};
          bool found = false;
          for (int32_t u = v0; u < v1 && !found; u += 32)
            found = __any_sync(0xffffffffu, fof_friends(a, G, T, p, a.rel[min(u + lane, v1 - 1)], D));
          if (found && lane == l) root = fof_union(a.group, pi, pk, a.status);
          __syncwarp();
        }
      }
    }
  }
}

// Octants of the queued cells, a warp each: the later octants of the cell and
// the octants or particles of the 13 neighbours, 32 at a time.  A lane looks at
// one of them (is it within reach, and another set?); those left are tested by
// the whole warp, pair by pair until the first friends.  300 us of the 1M
// clustered box, whatever the occupancy, the order of the nodes or the pairs
// tested: bound by the finds and unions that a core's octants contend in.
__global__ void __launch_bounds__(128) k_fof_link_octants(sphh::FofArgs a) {
  const GridDev G = a.grid[0];
  const int32_t nc = G.n_c;
  const FofTest T = fof_test(G, a.link);
  const float half = 0.5f * G.cell_f;
  const int lane = threadIdx.x & 31;
  const int64_t items = 8 * (int64_t)*a.queued;
  for (int64_t it = ((int64_t)blockIdx.x * blockDim.x + threadIdx.x) >> 5; it < items;
       it += ((int64_t)gridDim.x * blockDim.x) >> 5) {
    const int32_t cg = a.queue[it >> 3], c = cg - G.cell_base;
    const int me = (int)(it & 7);
    const int32_t own0 = a.cell_start[cg];
    const int32_t s0 = a.oct[own0 + me], s1 = me < 7 ? a.oct[own0 + me + 1] : a.cell_start[cg + 1];
    if (s0 >= s1) continue;
    const int32_t pm = __float_as_int(a.rel[s0].w);
    const float mx = me & 1 ? half : 0.0f, my = me & 2 ? half : 0.0f, mz = me & 4 ? half : 0.0f;
    const int32_t kx = c % nc, ky = (c / nc) % nc, kz = c / (nc * nc);
    int32_t root = fof_find<true>(a.group, pm, a.status);  // an ancestor of pm
    // lane o <= 13: cell o; its nodes (a dense one's octants, the particles of
    // another) follow those of the cells before it
    const FofCell M = lane <= kAxes ? fof_cell(a, G, kx, ky, kz, lane) : FofCell{0, 0, 0.f, 0.f, 0.f};
    int32_t incl = M.t1 - M.t0 >= kFofDense ? 8 : M.t1 - M.t0;
#pragma unroll
    for (int o = 1; o < 32; o <<= 1) {
      const int32_t v = __shfl_up_sync(0xffffffffu, incl, o);
      if (lane >= o) incl += v;
    }
    const int32_t nodes = __shfl_sync(0xffffffffu, incl, 31);
    for (int32_t n0 = 0; n0 < nodes; n0 += 32) {
      const int32_t n = n0 + lane;
      int o = 0;
#pragma unroll
      for (int step = 8; step > 0; step >>= 1)
        if (__shfl_sync(0xffffffffu, incl, o + step - 1) <= n) o += step;
      o = min(o, kAxes);
      const int32_t before = __shfl_sync(0xffffffffu, incl, max(o - 1, 0));
      const int k = n - (o > 0 ? before : 0);
      FofCell C;
      C.t0 = __shfl_sync(0xffffffffu, M.t0, o);
      C.t1 = __shfl_sync(0xffffffffu, M.t1, o);
      C.ox = __shfl_sync(0xffffffffu, M.ox, o);
      C.oy = __shfl_sync(0xffffffffu, M.oy, o);
      C.oz = __shfl_sync(0xffffffffu, M.oz, o);
      const bool dense = C.t1 - C.t0 >= kFofDense;  // at most kFofDense - 1 particles else
      int32_t u0 = 0, u1 = 0, pq = 0;
      bool open = n < nodes && (o > 0 || k > me);
      if (open) {
        u0 = dense ? a.oct[C.t0 + k] : C.t0 + k;
        u1 = dense ? (k < 7 ? a.oct[C.t0 + k + 1] : C.t1) : u0 + 1;
        open = u0 < u1;
      }
      if (open) {
        float gx, gy, gz;
        const float4 q = a.rel[u0];
        pq = __float_as_int(q.w);
        if (dense) {
          gx = fof_gap(mx, mx + half, C.ox, k & 1, half);
          gy = fof_gap(my, my + half, C.oy, (k >> 1) & 1, half);
          gz = fof_gap(mz, mz + half, C.oz, k >> 2, half);
        } else {
          gx = fof_gap(q.x + C.ox, q.x + C.ox, mx, 0, half);
          gy = fof_gap(q.y + C.oy, q.y + C.oy, my, 0, half);
          gz = fof_gap(q.z + C.oz, q.z + C.oz, mz, 0, half);
        }
        open = fmaf(gx, gx, fmaf(gy, gy, gz * gz)) < T.hi && !fof_joined(a.group, root, pq) &&
               fof_find<true>(a.group, pm, a.status) != fof_find<true>(a.group, pq, a.status);
      }
      for (unsigned left = __ballot_sync(0xffffffffu, open); left != 0u;) {
        const int l = __ffs((int)left) - 1;
        left &= left - 1u;
        const int32_t v0 = __shfl_sync(0xffffffffu, u0, l), v1 = __shfl_sync(0xffffffffu, u1, l);
        const FofCell D = {v0, v1, __shfl_sync(0xffffffffu, C.ox, l), __shfl_sync(0xffffffffu, C.oy, l),
                           __shfl_sync(0xffffffffu, C.oz, l)};
        // the other's box (an octant, or a particle)
        const bool dl = __shfl_sync(0xffffffffu, dense ? 1 : 0, l) != 0;
        const int kl = __shfl_sync(0xffffffffu, k, l);
        const float4 f = a.rel[v0];
        const float wx = D.ox + (dl ? (kl & 1 ? half : 0.0f) : f.x), wy = D.oy + (dl ? (kl & 2 ? half : 0.0f) : f.y),
                    wz = D.oz + (dl ? (kl & 4 ? half : 0.0f) : f.z), ww = dl ? half : 0.0f;
        // 32 of this octant's particles at a time against each of the other's
        bool found = false;
        for (int32_t s = s0; s < s1 && !found; s += 32) {
          const float4 p = a.rel[min(s + lane, s1 - 1)];
          // (those beside the other octant, or particle, only)
          const float px = fof_gap(p.x, p.x, wx, 0, ww), py = fof_gap(p.y, p.y, wy, 0, ww),
                      pz = fof_gap(p.z, p.z, wz, 0, ww);
          const bool near = fmaf(px, px, fmaf(py, py, pz * pz)) < T.hi;
          if (!__any_sync(0xffffffffu, near)) continue;
          for (int32_t u = v0; u < v1 && !found; u += 4) {
            bool hit = false;
#pragma unroll
            for (int i = 0; i < 4; ++i) hit = hit || (near && fof_friends(a, G, T, p, a.rel[min(u + i, v1 - 1)], D));
            found = __any_sync(0xffffffffu, hit);
          }
        }
        if (found) {
          if (lane == l) root = fof_union(a.group, pm, pq, a.status);
          root = __shfl_sync(0xffffffffu, root, l);
          // (the union may have taken in others of this batch)
          open = open && lane > l && fof_find<true>(a.group, pm, a.status) != fof_find<true>(a.group, pq, a.status);
          left = __ballot_sync(0xffffffffu, open);
        }
      }
    }
  }
}

// Final labels: every particle's root, the smallest index of its group.
__global__ void k_fof_label(sphh::FofArgs a) {
  for (int64_t p = (int64_t)blockIdx.x * blockDim.x + threadIdx.x; p < a.n_total;
       p += (int64_t)gridDim.x * blockDim.x)
    a.group[p] = fof_find<false>(a.group, (int32_t)p, a.status);
}

}  // namespace sphk

namespace sphh {
using namespace sphk;

cudaError_t launch_fof(const FofArgs& a, cudaStream_t st) {
  if (a.n_total <= 0) return cudaSuccess;
  int64_t b = (a.n_total + 255) / 256;
  if (b > 65535) b = 65535;
  cudaError_t e = cudaMemsetAsync(a.queued, 0, sizeof(int32_t), st);
  if (e != cudaSuccess) return e;
  k_fof_prep<<<(int)b, 256, 0, st>>>(a);
  k_fof_octants<<<a.num_sms * 8, 256, 0, st>>>(a);
  k_fof_link_octants<<<a.num_sms * 8, 128, 0, st>>>(a);
  k_fof_link<<<2 * (int)b, 128, 0, st>>>(a);
  k_fof_label<<<(int)b, 256, 0, st>>>(a);
  return cudaGetLastError();
}

}  // namespace sphh
