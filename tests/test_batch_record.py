"""The batch record of the neighbour search (csrc/batch_geometry.h), run on the CPU.

Asynchronous calls and graph replays read the staged record when they run, so calls on the
same batch must not disturb it while an earlier call's copy is pending.  A captured call keeps
its own candidate sweep and number of bins, so the record holds the bins of both sweeps.
"""
import ctypes
import os
import shutil
import subprocess

import numpy as np
import pytest

ROOT = os.path.dirname(os.path.dirname(os.path.abspath(__file__)))

DRIVER = r"""
#include <atomic>
#include <thread>
#include <vector>
#include "batch_geometry.h"

extern "C" int record_bytes(int S) { return (int)batch_record_bytes(S); }

// Stages the batch once, then `reps` times more while another thread reads the staged bytes as a
// pending copy would; returns how many of its reads differ from the first record.
extern "C" int differing_reads(const double* cell, const int64_t* offs, int S, double rc, int reps) {
  const size_t n = batch_record_bytes(S);
  std::vector<double> staged(n / 8), next(n / 8);
  BatchTotals t;
  if (stage_batch(cell, offs, S, rc, next.data(), staged.data(), &t) != BATCH_OK) return -1;
  const std::vector<double> first = staged;
  std::atomic<bool> stop{false};
  std::atomic<int> bad{0}, reads{0};
  std::thread reader([&] {
    while (!stop || reads < 100) {
      bad += std::memcmp(first.data(), staged.data(), n) != 0;
      ++reads;
    }
  });
  while (reads < 1) {}
  for (int k = 0; k < reps; ++k)
    if (stage_batch(cell, offs, S, rc, next.data(), staged.data(), &t) != BATCH_OK) bad += 1;
  stop = true;
  reader.join();
  return bad;
}

extern "C" int geometry(const double* cell, const int64_t* offs, int S, double rc, void* out, int* bins) {
  BatchTotals t;
  const int status = batch_geometry(cell, offs, S, rc, static_cast<StructGeom*>(out), &t);
  bins[0] = t.bins[0];
  bins[1] = t.bins[1];
  return status;
}
extern "C" int geom_bytes() { return (int)sizeof(StructGeom); }

// 1 if a batch that is refused leaves the staged record of the one before as it was
extern "C" int kept_by_a_refused_batch(const double* cell, const double* cell2, const int64_t* offs, int S, double rc) {
  const size_t n = batch_record_bytes(S);
  std::vector<double> staged(n / 8), next(n / 8);
  BatchTotals t;
  if (stage_batch(cell, offs, S, rc, next.data(), staged.data(), &t) != BATCH_OK) return -1;
  const std::vector<double> first = staged;
  if (stage_batch(cell2, offs, S, rc, next.data(), staged.data(), &t) == BATCH_OK) return -2;
  return std::memcmp(first.data(), staged.data(), n) == 0;
}
"""


@pytest.fixture(scope="module")
def lib(tmp_path_factory):
    cxx = os.environ.get("CXX") or shutil.which("g++")
    if cxx is None:
        pytest.skip("no C++ compiler")
    d = tmp_path_factory.mktemp("record")
    src, so = d / "driver.cpp", d / "driver.so"
    src.write_text(DRIVER)
    r = subprocess.run([cxx, "-std=c++17", "-O2", "-fPIC", "-shared", "-pthread", "-I",
                        os.path.join(ROOT, "paper_1905_02142_gb300", "csrc"), str(src), "-o", str(so)],
                       capture_output=True, text=True)
    assert r.returncode == 0, r.stderr
    out = ctypes.CDLL(str(so))
    p, i, d64 = ctypes.c_void_p, ctypes.c_int, ctypes.c_double
    out.differing_reads.argtypes = [p, p, i, d64, i]
    out.geometry.argtypes = [p, p, i, d64, p, p]
    out.kept_by_a_refused_batch.argtypes = [p, p, p, i, d64]
    return out


def batch(S, seed):
    """Cubes of 1 to 12 cutoffs an edge, with fewer and more than an atom per half-cutoff bin."""
    rng = np.random.default_rng(seed)
    edge = 4.0 * np.exp(rng.uniform(0.0, np.log(12.0), S))
    cell = np.eye(3)[None] * edge[:, None, None]
    cell[:, 1, 0] = 0.2 * edge * rng.random(S)
    n = (edge ** 3 * rng.uniform(0.01, 0.3, S)).astype(np.int64) + 1
    return np.ascontiguousarray(cell), np.concatenate([[0], np.cumsum(n)]).astype(np.int64)


@pytest.mark.parametrize("S", [1, 256])
def test_staging_the_same_batch_again_leaves_the_record_alone(lib, S):
    cell, offs = batch(S, 5)
    assert lib.differing_reads(cell.ctypes.data, offs.ctypes.data, S, 4.0, 2000) == 0


def test_refused_batch_leaves_the_record_alone(lib):
    cell, offs = batch(8, 6)
    for bad in (np.zeros((3, 3)), np.diag([0.02, 50.0, 50.0])):
        other = 1.1 * cell
        other[7] = bad
        assert lib.kept_by_a_refused_batch(cell.ctypes.data, other.ctypes.data, offs.ctypes.data, 8, 4.0) == 1


GRID = np.dtype([("nb", "i4", 3), ("m", "i4", 3), ("bin_off", "i4")])
GEOM = np.dtype([("h", "f8", (3, 3)), ("hinv", "f8", (3, 3)), ("h32", "f4", 9), ("h32lo", "f4", 9),
                 ("grid", GRID, 2), ("atom_off", "i4"), ("n_atoms", "i4"), ("margin", "f4")], align=True)


@pytest.mark.parametrize("S,rc", [(1, 4.0), (60, 4.0), (60, 5.3)])
def test_record_serves_either_sweep(lib, S, rc):
    """With the bins of its own sweep (number, offsets, ranges searched), as a captured call holds
    them, every atom's bin lies in its structure's range, the ranges fill the bins exactly, and
    two points within the cutoff are never further apart than the bins searched."""
    cell, offs = batch(S, 7)
    assert lib.geom_bytes() == GEOM.itemsize
    geom, bins = np.zeros(S, GEOM), np.zeros(2, np.int32)
    assert lib.geometry(cell.ctypes.data, offs.ctypes.data, S, rc, geom.ctypes.data, bins.ctypes.data) == 0
    assert np.array_equal(geom["h"], cell) and np.array_equal(geom["n_atoms"], np.diff(offs))
    assert bins[1] <= bins[0] + offs[-1]        # what the bin buffers are sized for
    rng = np.random.default_rng(8)
    differ = 0
    for w in (0, 1):
        end = 0
        for s in range(S):
            g = geom["grid"][s, w]
            assert g["bin_off"] == end
            end += int(np.prod(g["nb"]))
            f = rng.random((400, 3))
            f[:8] = np.array(np.meshgrid(*[[0.0, 1 - 1e-12]] * 3)).reshape(3, -1).T
            step = rng.normal(size=(400, 3))
            step *= rc * np.minimum(1.0, rng.uniform(0.9, 1.02, (400, 1))) / np.linalg.norm(step, axis=1, keepdims=True)
            here = np.minimum(np.floor(f * g["nb"]).astype(int), g["nb"] - 1)
            there = np.floor((f + step @ geom["hinv"][s]) * g["nb"]).astype(int)
            assert (np.abs(there - here) <= g["m"]).all()
            bin_id = g["bin_off"] + (here[:, 0] * g["nb"][1] + here[:, 1]) * g["nb"][2] + here[:, 2]
            assert bin_id.min() >= g["bin_off"] and bin_id.max() < end
            differ += w == 1 and int(np.prod(g["nb"])) > int(np.prod(geom["grid"][s, 0]["nb"]))
        assert end == bins[w]
    assert differ > 0                           # narrow bins were among them
