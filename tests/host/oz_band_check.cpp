// Host check of the band order in csrc/oz_order.cuh: for full and lower C, tile
// grids up to 60 x 60 and bands of 1 .. 16 and 4096 tile rows, the items
// 0 .. oz_item_count - 1 name every output tile exactly once (for a lower C those
// with tm >= tn) and no other; a band of one row is the row-by-row order.
#include <cstdio>
#include <vector>

#include OZ_ORDER_HEADER

using namespace qmlgb;

static int check(int tiles_m, int tiles_n, int lower, int band) {
  std::vector<int> hit((size_t)tiles_m * tiles_n, 0);
  const int count = oz_item_count(tiles_m, tiles_n, lower, 0);
  for (int i = 0; i < count; ++i) {
    int tm = -1, tn = -1, rm, rn;
    oz_band_tile_of(tiles_m, tiles_n, lower, band, i, tm, tn);
    oz_tile_of(lower, tiles_n, i, rm, rn);
    const bool in = tm >= 0 && tm < tiles_m && tn >= 0 && tn < tiles_n && !(lower && tn > tm);
    if (!in || hit[(size_t)tm * tiles_n + tn]++ || (band == 1 && (tm != rm || tn != rn))) {
      std::printf("FAIL tiles=%dx%d lower=%d band=%d item=%d\n", tiles_m, tiles_n, lower, band, i);
      return 1;
    }
  }
  return 0;  // count distinct tiles of the output: all of them
}

int main() {
  for (int lower = 0; lower < 2; ++lower)
    for (int tiles_m = 1; tiles_m <= 60; ++tiles_m)
      for (int tiles_n = 1; tiles_n <= 60; ++tiles_n)
        for (int band : {1, 2, 3, 5, 8, 12, 16, 4096})
          if (!(lower && tiles_n != tiles_m) && check(tiles_m, tiles_n, lower, band)) return 1;
  std::printf("OK\n");
  return 0;
}
