// The launchers of csrc/ on one device after another (linked with fake_cuda.cpp:
// no kernel runs).  Prints "<launcher> <device> <status>".
#include <cstdio>

#include "../../paper_2305_13380_gb300/csrc/sph_internal.cuh"
#include "../../paper_2305_13380_gb300/csrc/sph_launch.h"
#include "../../paper_2305_13380_gb300/csrc/tree.cuh"

extern int fake_device;

int main() {
  using namespace sphh;
  sphk::PhysDev ph{};
  const sphk::SphenixDev sx;
  static float4 four[1];
  static int32_t words[64];
  for (int device : {0, 1, 0, 2, 63, 64, 65}) {
    fake_device = device;
    auto report = [&](const char* name, cudaError_t e) { std::printf("%s %d %d\n", name, device, (int)e); };
    static uint64_t keys[8];
    static int8_t levels[8];
    report("radix_sort_index", radix_sort_index(5000, 20, words, words, words, words, words, words, nullptr));
    report("radix_sort_index64", radix_sort_index64(8192, 50, keys, keys, keys, words, words, words, nullptr));
    report("radix_partition", radix_partition(100, levels, words, words, nullptr));
    for (int k = 0; k < sphk::kNumKernels; ++k) {
      ph.kernel = k;
      DensityArgs d{};
      d.num_sms = 152;
      d.misc = words;
      report("launch_density", launch_density(d, ph, nullptr));
      ForceArgs f{};
      f.num_sms = 152;
      f.misc = words;
      f.fE = four;
      f.alpha_c_out = (float*)words;
      f.bins_out = words;
      report("launch_force", launch_force(f, ph, nullptr));
      report("launch_sphenix_force", launch_sphenix_force(f, ph, sx, nullptr));
      report("launch_sphenix_gradient", launch_sphenix_gradient(f, ph, sx, nullptr));
      report("launch_limit_bins", launch_limit_bins(f, ph, nullptr));
      TreeDensityArgs t{};
      t.num_sms = 152;
      t.n_total = 10000;
      report("launch_tree_density", launch_tree_density(t, ph, nullptr));
      t.act = (const uint8_t*)words;
      report("launch_tree_density(masked)", launch_tree_density(t, ph, nullptr));
      TreeForceArgs g{};
      g.num_sms = 152;
      g.n_total = 10000;
      report("launch_tree_force", launch_tree_force(g, ph, nullptr));
    }
    ForceArgs f{};
    f.num_sms = 152;
    SymArgs y{};
    report("launch_force_sym", launch_force_sym(f, y, ph, 5000, nullptr));
  }
  return 0;
}
