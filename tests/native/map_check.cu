// Host-side check of map_index: for every axis length, boundary pair and position that the
// 32-wide, up to 16-row tiles and their halos can ask for, the answer is a cell of the axis;
// positions within two cells of a side (the stencils' reach) map as the boundary says.
#include <cstdio>

#include "m2c_kernels.cuh"

int main() {
  long long outside = 0, wrong = 0;
  const int T = M2C_BC_TRANSMISSIVE, P = M2C_BC_PERIODIC, S = M2C_BC_SYMMETRY;
  const int pairs[5][2] = {{T, T}, {P, P}, {S, T}, {T, S}, {S, S}};
  for (int n = 1; n <= 80; ++n)
    for (auto& b : pairs) {
      if (n < 2 && (b[0] == S || b[1] == S)) continue;  // refused by the grid's checks
      for (int i = -2; i < (n + 31) / 32 * 32 + 2; ++i) {
        const int m = m2c::map_index(i, n, b[0], b[1]);
        outside += m < 0 || m >= n;
        if (i >= n + 2) continue;
        int want = i;
        if (i < 0) want = b[0] == T ? 0 : b[0] == S ? -1 - i : ((i % n) + n) % n;
        if (i >= n) want = b[1] == T ? n - 1 : b[1] == S ? 2 * n - 1 - i : i % n;
        wrong += m != want;
      }
    }
  std::printf("positions outside %lld wrong %lld\n", outside, wrong);
  return outside || wrong ? 1 : 0;
}
