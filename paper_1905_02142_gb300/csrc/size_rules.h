// Rules that pick a tile or a capacity from a call's sizes, in plain C++ (no CUDA) so that tests
// run them on the CPU over sizes that no test would launch.
#pragma once

#include <stddef.h>

#include <algorithm>

#ifdef __CUDACC__
#define SG_HOST_DEVICE __host__ __device__
#else
#define SG_HOST_DEVICE
#endif

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

// Channel row of the power spectrum in shared memory, in elements of `elem` bytes: L of them padded
// to an odd number of 16-byte steps, so that rows start in different banks.
SG_HOST_DEVICE constexpr int powspec_row(int L, int elem) { return ((L * elem + 15) / 16 | 1) * (16 / elem); }

// Warps per block of the power spectrum (one atom each) and the elements of one warp's region
// (channel rows, then p); 0 warps where the descriptor is too large.  The limit and the warps
// follow the data, 200 KB of it at most; the rows' padding comes on top, up to 202.2 KB in all over
// every basis and species count, within a block's 227 KB.
struct PowspecShape { int warps, per_warp; };
inline PowspecShape powspec_shape(int nch, int lmax, int elem) {
  const int L = (lmax + 1) * (lmax + 1), D = nch * (nch + 1) / 2 * (lmax + 1);
  const size_t data = (size_t)((nch * L + D + 3) / 4 * 4) * elem;
  return {(int)std::min<size_t>(4, 200 * 1024 / data), (nch * powspec_row(L, elem) + D + 3) / 4 * 4};
}

// Neighbour slots per atom of a batch whose largest neighbour count `most` has been measured: room
// for a few more, in steps of 8.
inline int measured_slots(int most) { return (most + 8 + 7) & ~7; }

// Slots that the next call on a batch of this shape takes: what this configuration measured, at
// least the estimate from the densities `est`, at most the `used` ones whose buffers are there.  A
// call that took more because the configuration before it was denser lets them go again (they
// cost placement its shared memory); one that needed more than the estimate keeps its room of 8,
// so that counts around the estimate do not overflow at every other call.
inline int slots_after(int est, int most, int used) { return std::min(used, std::max(est, measured_slots(most))); }
