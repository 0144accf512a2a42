// zero_runs.cpp -- test harness: the runs of nodes outside the mask cover them
// all once, in pieces short enough for warps to share evenly.  Built and run by
// tests/test_zero_runs.py; the GPU solver's entry points are stubbed.
#include <cstdio>
#include <random>
#include <string>
#include <vector>

#include "table.h"

namespace patbp {
struct GpuEikonal {};
GpuEikonal* gpu_eikonal_create(const GridDesc&, const float*, const std::vector<int32_t>&, int, std::string&) {
  return nullptr;
}
bool gpu_eikonal_slot_times(GpuEikonal*, const double*, int, double, double*, std::string&) { return false; }
void gpu_eikonal_destroy(GpuEikonal*) {}
int gpu_eikonal_batch(const GridDesc&, int64_t, size_t) { return 1; }
}  // namespace patbp

using namespace patbp;

int main() {
  std::mt19937 rng(1);
  const double sensors[6] = {0.0, 0.0, 0.0, 1e-3, 2e-3, 0.0};
  for (int kind = 0; kind < 6; ++kind) {
    GridDesc g;
    g.ndim = 2;
    g.n[0] = 130;
    g.n[1] = 97;
    g.n[2] = 1;
    g.dx = 1e-4;
    const int64_t n = g.total();
    std::vector<uint8_t> mask(static_cast<size_t>(n), 0);
    for (int64_t v = 0; v < n; ++v)
      mask[size_t(v)] = kind == 0 ? v == n - 1 : kind == 1 ? v == 0 : kind == 2 ? (rng() & 1) : kind == 3 ? 1
                        : kind == 4 ? v % 513 == 512 : v % 1025 == 7;
    HostTable t;
    std::string err;
    if (!build_constant_layout(1500.0, g, sensors, 2, mask.data(), 2e-8, 1000, 128, false, t, err)) {
      std::printf("layout: %s\n", err.c_str());
      return 1;
    }
    std::vector<int> hit(static_cast<size_t>(n), 0);
    for (size_t r = 0; r < t.zero_runs.size(); r += 2) {
      const int64_t at = t.zero_runs[r], len = t.zero_runs[r + 1];
      if (len < 1 || len > 512 || at < 0 || at + len > n) {
        std::printf("kind %d: run of %lld nodes at %lld\n", kind, (long long)len, (long long)at);
        return 1;
      }
      for (int64_t v = at; v < at + len; ++v) hit[size_t(v)]++;
    }
    for (int64_t v = 0; v < n; ++v)
      if (hit[size_t(v)] != (mask[size_t(v)] ? 0 : 1)) {
        std::printf("kind %d: node %lld\n", kind, (long long)v);
        return 1;
      }
  }
  std::printf("ok\n");
  return 0;
}
