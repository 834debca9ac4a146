// Parts of the library behind its entry points, for the tests that drive them
// directly (linked with libsph.so).
#include "../../paper_2305_13380_gb300/csrc/sph_internal.cuh"
#include "../../paper_2305_13380_gb300/csrc/sph_launch.h"
#include "../../paper_2305_13380_gb300/csrc/tree.cuh"

// The fine coordinate of each x by the estimate (or the exact path, where the estimate
// leaves it to that) and by the definition, in a box of side L of n_c cells.
__global__ void k_fine_coords(long n, const double* x, double L, int n_c, int32_t* fast, int32_t* exact) {
  sphk::GridDev G;
  G.L = L;
  G.n_c = n_c;
  G.fine_scale = (double)n_c * (double)sphk::kTreeFine / L;
  for (long i = (long)blockIdx.x * blockDim.x + threadIdx.x; i < n; i += (long)gridDim.x * blockDim.x) {
    const int32_t k = sphk::cell_coord(x[i], L, n_c);
    fast[i] = sphk::fine_coord_fast(x[i], G, k);
    exact[i] = sphk::fine_coord(x[i], L, n_c, k);
  }
}

extern "C" {

long part_scan_words(long n) { return sphh::scan_words(n); }
int part_scan(const int32_t* in, int32_t* out, long n, int32_t* scratch, cudaStream_t st) {
  return (int)sphh::scan_exclusive(in, out, n, scratch, 152, st);
}
int part_scan_bytes(const uint8_t* in, int32_t* out, long n, int32_t* scratch, cudaStream_t st) {
  return (int)sphh::scan_exclusive(in, out, n, scratch, 152, st);
}
int part_sort_reverse_pairs(long n, const int32_t* start, uint32_t* rev, int32_t* queue, int32_t* counts,
                            cudaStream_t st) {
  return (int)sphh::sort_reverse_pairs(n, start, rev, queue, counts, counts + 1, 152, st);
}
int part_fine_coords(long n, const double* x, double L, int n_c, int32_t* fast, int32_t* exact, cudaStream_t st) {
  k_fine_coords<<<256, 256, 0, st>>>(n, x, L, n_c, fast, exact);
  return (int)cudaGetLastError();
}

}
