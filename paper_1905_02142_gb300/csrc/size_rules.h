// Rules that pick a tile or a capacity from a call's sizes, in plain C++ (no CUDA) so that tests
// run them on the CPU over sizes that no test would launch.
#pragma once

// Tile of an n x m FP64 product on CUDA cores over `sms` SMs: the one whose busiest SM has the
// fewest elements (the larger tile when equal: fewer loads per element).  Row tiles lie on
// gridDim.y, which ends at 65535: 32-row tiles stop at 2,097,120 rows, 64-row ones at 4,194,240.
struct SimtTile { int m, n; };
inline SimtTile simt_tile_f64(int n, int m, int sms) {
  constexpr SimtTile tiles[3] = {{64, 64}, {32, 32}, {32, 16}};
  constexpr long long GRID_Y = 65535;
  SimtTile best = tiles[0];
  long long best_cost = -1;
  for (const SimtTile& t : tiles) {
    const long long rows = ((long long)n + t.m - 1) / t.m;
    if (rows > GRID_Y) continue;
    const long long count = rows * (((long long)m + t.n - 1) / t.n);
    const long long cost = (count + sms - 1) / sms * t.m * t.n;
    if (best_cost < 0 || cost < best_cost) {
      best = t;
      best_cost = cost;
    }
  }
  return best;
}
