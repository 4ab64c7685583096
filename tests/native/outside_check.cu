// Host-side check of the bulk kernel's cells outside a tile: whichever cell a lane of the
// last three warps takes, its slot of the shared plane and both neighbours' are slots that
// the plane loop writes (the own rows up to one beyond the grid's last, and the halo ring),
// for tiles cut by the grid's edge after any number of rows. Prints the count of misses.
#include <cstdio>
#include <vector>

#include "m2c_stage.cuh"

template <int TY>
static int check() {
  constexpr int TX = 32, HX = TX + 4, HY = TY + 4, NHALO = (4 * TY + 31) / 32 * 32 + 4 * TX;
  int misses = 0;
  for (int rows = 1; rows <= TY; ++rows) {  // rows of the tile inside the grid
    std::vector<char> written(HX * HY, 0);
    for (int ty = 0; ty < TY; ++ty)
      if (ty <= rows + 1)
        for (int tx = 0; tx < TX; ++tx) written[(ty + 2) * HX + tx + 2] = 1;
    for (int h = 0; h < NHALO; ++h) {
      const int s = m2c::halo_slot_of<TY>(h);
      if (s >= 0) written[s] = 1;
    }
    for (int ty = TY - 3; ty < TY; ++ty) {
      if (ty == TY - 1 && rows < TY) continue;  // row TY is not taken (one beyond the grid at least)
      for (int tx = 0; tx < TX; ++tx)
        for (int on = 0; on < 2; ++on) {
          // the lanes that a cell counts for; the others of the x warp run with on = false
          if (on && ty == TY - 3 && (tx / TY >= 2 || (tx & (TY - 1)) >= rows)) continue;
          int so = 0;
          const int c = m2c::outside_slot<TY>(ty, tx, on != 0, so);
          for (int d = -1; d <= 1; ++d) {
            const int s = c + d * so;
            if (s < 0 || s >= HX * HY || !written[s]) {
              if (misses++ < 5) std::printf("rows %d of %d, warp %d lane %d on %d: slot %d\n", rows, TY, ty, tx, on, s);
            }
          }
        }
    }
  }
  return misses;
}

int main() {
  const int misses = check<4>() + check<8>() + check<16>();
  std::printf("unwritten slots read %d\n", misses);
  return misses ? 1 : 0;
}
