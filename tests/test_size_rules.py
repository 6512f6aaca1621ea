"""Rules that pick a tile or a capacity from a call's sizes (csrc/size_rules.h), run on the CPU
at sizes that no test launches."""
import ctypes
import os
import shutil
import subprocess

import pytest

ROOT = os.path.dirname(os.path.dirname(os.path.abspath(__file__)))

DRIVER = r"""
#include "size_rules.h"
extern "C" void tile_f64(int n, int m, int sms, int* out) {
  const SimtTile t = simt_tile_f64(n, m, sms);
  out[0] = t.m;
  out[1] = t.n;
}
extern "C" int slots(int est, int most, int used) { return slots_after(est, most, used); }
extern "C" int measured(int most) { return measured_slots(most); }
extern "C" void powspec(int nch, int lmax, int elem, int* out) {
  const PowspecShape y = powspec_shape(nch, lmax, elem);
  out[0] = y.warps;
  out[1] = y.per_warp;
  out[2] = powspec_row((lmax + 1) * (lmax + 1), elem);
}
"""

GRID_Y = 65535


@pytest.fixture(scope="module")
def lib(tmp_path_factory):
    cxx = os.environ.get("CXX") or shutil.which("g++")
    if cxx is None:
        pytest.skip("no C++ compiler")
    d = tmp_path_factory.mktemp("rules")
    src, so = d / "driver.cpp", d / "driver.so"
    src.write_text(DRIVER)
    r = subprocess.run([cxx, "-std=c++17", "-O2", "-fPIC", "-shared", "-I",
                        os.path.join(ROOT, "paper_1905_02142_gb300", "csrc"), str(src), "-o", str(so)],
                       capture_output=True, text=True)
    assert r.returncode == 0, r.stderr
    return ctypes.CDLL(str(so))


def tile_f64(lib, n, m, sms=152):
    out = (ctypes.c_int * 2)()
    lib.tile_f64(n, m, sms, out)
    return tuple(out)


def cost(tile, n, m, sms=152):
    rows, cols = -(-n // tile[0]), -(-m // tile[1])
    return -(-rows * cols // sms) * tile[0] * tile[1]


@pytest.mark.parametrize("m", [1, 16, 17, 32, 33, 64, 65, 100, 324, 500, 605, 4096])
@pytest.mark.parametrize("n", [1, 32, 33, 1000, 100_000, 2_097_119, 2_097_120, 2_097_121, 3_000_000, 4_194_239,
                               4_194_240])
def test_fp64_tiles_fit_the_launch_grid(lib, n, m):
    """The tile with the least work for the busiest SM among those whose row blocks a grid holds:
    every size up to 65535 rows of 64-row blocks can be launched."""
    t = tile_f64(lib, n, m)
    assert -(-n // t[0]) <= GRID_Y
    fit = [c for c in ((64, 64), (32, 32), (32, 16)) if -(-n // c[0]) <= GRID_Y]
    assert cost(t, n, m) == min(cost(c, n, m) for c in fit)


def test_fp64_tiles_beyond_the_grid_stay_refused(lib):
    assert tile_f64(lib, 4_194_241, 100) == (64, 64)


@pytest.mark.parametrize("elem", [4, 8])
def test_power_spectrum_blocks_fit_shared_memory(lib, elem):
    """Every basis and species count whose unpadded rows fit 200 KB runs, with as many warps per
    block as those rows allow, and with its padded rows within a block's 227 KB."""
    out = (ctypes.c_int * 3)()
    refused = 0
    for nsp in range(1, 9):
        for n_max in range(2, 13):
            for l_max in range(13):
                nch, L = nsp * n_max, (l_max + 1) ** 2
                data = -(-(nch * L + nch * (nch + 1) // 2 * (l_max + 1)) // 4) * 4 * elem
                lib.powspec(nch, l_max, elem, out)
                warps, per_warp, row = out
                assert warps == min(4, 200 * 1024 // data), (nsp, n_max, l_max)
                assert warps * per_warp * elem <= 227 * 1024
                assert per_warp % 4 == 0 and per_warp >= nch * row + nch * (nch + 1) // 2 * (l_max + 1)
                assert row >= L and row * elem % 16 == 0 and row * elem // 16 % 2 == 1
                refused += warps == 0
    assert refused > 0


def test_neighbour_slots_follow_the_configuration(lib):
    """Slots of a run of calls that each take what the one before left (at least the estimate): a
    dense configuration raises them, a sparser one lets them fall back to the estimate at once, and
    counts that fluctuate around the estimate never overflow after the first."""
    est = 80

    def calls(counts, slots):
        overflows = 0
        for most in counts:
            used = max(est, slots)
            if most > used:                      # repeated at the measured size
                overflows += 1
                used = lib.measured(most)
                slots = used
            else:
                slots = lib.slots(est, most, used)
            assert most <= slots <= used
        return slots, overflows

    assert calls([40, 60, 75], est) == (est, 0)
    dense, n = calls([300], est)
    assert dense >= 300 and n == 1
    assert calls([41], dense) == (est, 0)        # a sparse configuration after a dense one
    slots, n = calls([290, 297, 299, 300], dense)
    assert n == 0 and 300 <= slots <= dense
    slots, n = calls([81, 79, 82, 78, 81, 80, 85, 77, 85], est)
    assert n == 1 and slots <= 96
