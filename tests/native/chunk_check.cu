// Host-side check of chunk_planes: a requested chunk length is kept, an automatic one gives
// the same number of chunks with lengths that differ by at most one plane on average.
#include <cstdio>

#include "m2c_stage.h"

int main() {
  int wrong = 0;
  for (int nz = 1; nz <= 300; ++nz)
    for (int tz = 1; tz <= 80; ++tz) {
      const int want = tz < nz ? tz : nz, chunks = (nz + want - 1) / want;
      wrong += m2c::chunk_planes(nz, tz, true) != want;
      const int a = m2c::chunk_planes(nz, tz, false);
      wrong += a < 1 || a > want || (nz + a - 1) / a != chunks || a != (nz + chunks - 1) / chunks;
    }
  std::printf("wrong chunks %d\n", wrong);
  return wrong ? 1 : 0;
}
