// Parts of the library behind its entry points, for the tests that drive them
// directly (linked with libsph.so).
#include "../../paper_2305_13380_gb300/csrc/sph_internal.cuh"
#include "../../paper_2305_13380_gb300/csrc/sph_launch.h"

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

}
