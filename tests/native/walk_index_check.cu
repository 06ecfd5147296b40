// Host-side check of walk_index_fits (air_internal.cuh): for uniform grids around
// 2^31 cells and every chunk length of the walk, wherever 32-bit indices are
// chosen, no index that a ray's walk forms, K planes beyond the grid included,
// leaves the range of a 32-bit integer; and small grids keep 32-bit indices.
// Prints "ok <cases>" and exits 0, or the first mismatch and exits 1.
#include <cstdint>
#include <cstdio>
#include <initializer_list>

#include "air_internal.cuh"

int main() {
  long long cases = 0, chosen = 0;
  const int side[][2] = {{1000, 1000}, {1290, 1290}, {46340, 46340}, {1, 1}, {2048, 512}, {33, 77}};
  for (const auto &s : side)
    for (int K : {4, 8, 16}) {
      const int64_t plane = (int64_t)s[0] * s[1];
      const int64_t top = 0x7fffffffLL / plane;
      for (int64_t n2 = top - 40 > 1 ? top - 40 : 1; n2 <= top + 2 && n2 < 0x7fffffff; ++n2, ++cases) {
        if (!air::walk_index_fits(s[0], s[1], (int)n2, K)) continue;
        ++chosen;
        // from the last cell on along +z, and from the first along -z
        int64_t up = plane * n2 - 1, down = 0;
        for (int u = 0; u < K; ++u) {
          up += plane;
          down -= plane;
        }
        if (up > INT32_MAX || down < INT32_MIN) {
          std::printf("%d x %d x %lld, K %d: index %lld\n", s[0], s[1], (long long)n2, K, (long long)up);
          return 1;
        }
      }
    }
  if (!chosen || !air::walk_index_fits(512, 512, 512, 16)) {
    std::printf("32-bit indices refused\n");
    return 1;
  }
  std::printf("ok %lld\n", cases);
  return 0;
}
