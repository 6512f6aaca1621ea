// The batch record of the neighbour search, built on the host in FP64: the geometry of every
// structure, followed by the atom offsets.  One copy takes it to the device, through pinned
// staging that asynchronous calls and graph replays read when they run, not when they are
// queued.  It therefore depends on the batch and the list radius alone (it holds the bins of
// both candidate sweeps, and the launches that were queued or captured say which they use), is
// built beside the staging and replaces what is there only where it differs: a call on the
// same batch leaves the staged bytes alone, whatever its tile plan and whatever copies are
// pending, and so does a batch that is refused.  Plain C++ (no CUDA), so that tests run it on
// the CPU.
#pragma once

#include <stdint.h>

#include <algorithm>
#include <cmath>
#include <cstring>

// Bins of one structure.
struct BinGrid {
  int nb[3];       // bins along each lattice direction
  int m[3];        // bin offsets searched: -m..m
  int bin_off;     // first bin of this structure in the flattened bin arrays
};

// Per-structure geometry for the neighbour builder.
struct StructGeom {
  double h[9];     // rows = lattice vectors
  double hinv[9];  // inverse (fractional = x @ hinv)
  float h32[9];
  float h32lo[9];  // h - (double)h32, so that h = h32 + h32lo to ~2^-48
  BinGrid grid[2]; // of the sweep by bin (bins at least r_cut wide), and of the sweep by atom
  int atom_off, n_atoms;
  float margin;    // |d2_fp32 - rc^2| below which the FP64 test decides
};

inline size_t batch_record_bytes(int S) { return sizeof(StructGeom) * (size_t)S + sizeof(int64_t) * (size_t)(S + 1); }
static_assert(sizeof(StructGeom) % alignof(int64_t) == 0, "the atom offsets follow the geometry");

// distance between the lattice planes of direction k of cell c
inline double plane_distance(const double* c, int k) {
  const double* u = c + 3 * ((k + 1) % 3);
  const double* v = c + 3 * ((k + 2) % 3);
  const double cx = u[1] * v[2] - u[2] * v[1], cy = u[2] * v[0] - u[0] * v[2], cz = u[0] * v[1] - u[1] * v[0];
  const double det = c[0] * (c[4] * c[8] - c[5] * c[7]) - c[1] * (c[3] * c[8] - c[5] * c[6]) +
                     c[2] * (c[3] * c[7] - c[4] * c[6]);
  return std::fabs(det) / std::sqrt(cx * cx + cy * cy + cz * cz);
}

enum BatchStatus { BATCH_OK = 0, BATCH_SINGULAR, BATCH_THIN };
struct BatchTotals {
  int bins[2];       // of each grid
  int max_atoms;
  double slot_est;   // pairs per atom of the densest structure
  int failed;        // the structure of a status other than BATCH_OK
};

// Geometry of a batch: cell [S][9], offs [S + 1], rc the list radius.
// A sweep by atom reads its candidates bin by bin for every atom, so its bins are half the cutoff
// wide: 125 of them around an atom hold 58 % of the volume of 27 wide ones (1000 atoms 18.0 ->
// 13.2 us, 10,000 atoms 34.2 -> 28.3 us, the 256-structure batch 376 -> 238 us).  Structures with less
// than an atom per narrow bin keep the wide ones: there the sweep is a walk over bins, not over
// atoms.
inline BatchStatus batch_geometry(const double* cell, const int64_t* offs, int S, double rc, StructGeom* out,
                                  BatchTotals* t) {
  std::memset(static_cast<void*>(out), 0, sizeof(StructGeom) * (size_t)S);
  *t = BatchTotals{};
  for (int s = 0; s < S; ++s) {
    StructGeom& g = out[s];
    const double* c = cell + 9 * s;
    for (int k = 0; k < 9; ++k) {
      g.h[k] = c[k];
      g.h32[k] = (float)c[k];
      g.h32lo[k] = (float)(c[k] - (double)g.h32[k]);
    }
    const double det = c[0] * (c[4] * c[8] - c[5] * c[7]) - c[1] * (c[3] * c[8] - c[5] * c[6]) +
                       c[2] * (c[3] * c[7] - c[4] * c[6]);
    t->failed = s;
    if (!(std::fabs(det) > 0) || !std::isfinite(det)) return BATCH_SINGULAR;
    // inverse (rows of h are lattice vectors; fractional = x @ hinv)
    double inv[9] = {c[4] * c[8] - c[5] * c[7], c[2] * c[7] - c[1] * c[8], c[1] * c[5] - c[2] * c[4],
                     c[5] * c[6] - c[3] * c[8], c[0] * c[8] - c[2] * c[6], c[2] * c[3] - c[0] * c[5],
                     c[3] * c[7] - c[4] * c[6], c[1] * c[6] - c[0] * c[7], c[0] * c[4] - c[1] * c[3]};
    for (int k = 0; k < 9; ++k) g.hinv[k] = inv[k] / det;
    const int na = (int)(offs[s + 1] - offs[s]);
    double H = 0, dk[3];
    int mmax = 0, nb2[3];
    BinGrid &wide = g.grid[0], &narrow = g.grid[1];
    for (int k = 0; k < 3; ++k) {
      dk[k] = plane_distance(c, k);
      int nb = (int)std::floor(dk[k] / rc);
      if (nb < 1) nb = 1;
      const int nb_cap = std::max(1, (int)std::cbrt((double)std::max(na, 1)) + 1);
      if (nb > 2 * nb_cap) nb = 2 * nb_cap;  // no more bins than atoms need
      wide.nb[k] = nb;
      wide.m[k] = (int)std::floor(rc * nb / dk[k]) + 1;
      if (wide.m[k] > 100) return BATCH_THIN;
      mmax = std::max(mmax, wide.m[k]);
      nb2[k] = std::max(nb, (int)std::min(std::floor(2.0 * dk[k] / rc), 2.0 * nb + 1.0));
      H += std::sqrt(c[3 * k] * c[3 * k] + c[3 * k + 1] * c[3 * k + 1] + c[3 * k + 2] * c[3 * k + 2]);
    }
    const double X = H * (mmax + 3), u = std::ldexp(1.0, -24);
    // |error| of each FP32 separation component <= 10 u X (rounded positions, FP32 shift from
    // rounded lattice vectors, two additions); the margin bounds the error of d2 twice over
    g.margin = (float)(2.0 * (2.0 * std::sqrt(3.0) * 10.0 * rc * X * u + 4.0 * rc * rc * u) + 1e-30);
    t->max_atoms = std::max(t->max_atoms, na);
    // kept pairs per atom ~ density x sphere volume (periodic images included)
    t->slot_est = std::max(t->slot_est, (double)na / std::fabs(det) * 4.18879020478639 * rc * rc * rc);
    g.atom_off = (int)offs[s];
    g.n_atoms = na;
    narrow = wide;
    if ((long long)nb2[0] * nb2[1] * nb2[2] <= na)
      for (int k = 0; k < 3; ++k) {
        narrow.nb[k] = nb2[k];
        narrow.m[k] = (int)std::floor(rc * nb2[k] / dk[k]) + 1;
      }
    for (int w = 0; w < 2; ++w) {
      g.grid[w].bin_off = t->bins[w];
      t->bins[w] += g.grid[w].nb[0] * g.grid[w].nb[1] * g.grid[w].nb[2];
    }
  }
  return BATCH_OK;
}

// The whole record of a batch into `next` (batch_record_bytes(S) bytes, 8-byte aligned) and from
// there to `staged`, if the bytes differ.
inline BatchStatus stage_batch(const double* cell, const int64_t* offs, int S, double rc, void* next, void* staged,
                               BatchTotals* t) {
  StructGeom* const g = static_cast<StructGeom*>(next);
  const BatchStatus status = batch_geometry(cell, offs, S, rc, g, t);
  if (status != BATCH_OK) return status;
  std::memcpy(static_cast<void*>(g + S), offs, sizeof(int64_t) * (size_t)(S + 1));
  if (std::memcmp(staged, next, batch_record_bytes(S)) != 0) std::memcpy(staged, next, batch_record_bytes(S));
  return BATCH_OK;
}
