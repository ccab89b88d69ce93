"""The parts of the CUDA path's headers that compile for the host too, built with
g++ and checked without a GPU."""

import os
import subprocess

import pytest

ROOT = os.path.dirname(os.path.dirname(os.path.abspath(__file__)))
CSRC = os.path.join(ROOT, "paper_2109_01329_gb300", "csrc")
INCLUDE = os.path.join(ROOT, "include")


def _build(path, code, *flags):
    """Compiles C++ source text against the headers; the path of what it makes."""
    src, out = str(path / "t.cpp"), str(path / "t.bin")
    with open(src, "w") as f:
        f.write(code)
    subprocess.run(["g++", "-std=c++17", "-O2", "-ffp-contract=off", "-I", CSRC, "-I", INCLUDE, src, "-o", out, *flags],
                   check=True, timeout=300)
    return out


def test_jump_table_is_aligned_for_16_byte_loads(tmp_path):
    """The kernels read the table of jump matrices in 16-byte pieces: the type, not
    the order in which a linker lays globals, has to place every row and second
    matrix on such a boundary."""
    exe = _build(tmp_path, """
#include <cstdio>
#include "mrg_tables.h"
int main() { std::printf("%zu %zu", alignof(grng::mrg::DigitTable), sizeof(grng::mrg::DigitTable::row[0])); }
""")
    align, row = map(int, subprocess.run([exe], check=True, capture_output=True, text=True).stdout.split())
    assert align % 16 == 0 and row % 16 == 0


def test_batch_launch_count_heals_after_overlaps(tmp_path):
    """CTAs of up to three launches of one batch arriving in any order: a launch
    that runs alone shows one count to all of its CTAs, and once launches that
    overlapped are over the count is their number, exactly."""
    exe = _build(tmp_path, """
#include <algorithm>
#include <cstdio>
#include <random>
#include <vector>
#include "grng_internal.h"
using namespace grng;
int main() {
  std::mt19937 r(7);
  uint64_t arrivals = 0, launches = 0;
  const uint32_t grids[] = {1, 2, 3, 152, 4864, 1u << kArrivalBits};
  for (int trial = 0; trial < 300; ++trial) {
    std::vector<uint64_t> shares;  // what the CTAs of this trial's launches add
    const int k = trial % 3 + 1;
    for (int i = 0; i < k; ++i) {
      const uint32_t ctas = grids[r() % (trial < 6 ? 6 : 5)];
      for (uint32_t c = 0; c < ctas; ++c) shares.push_back(batch_arrival(c, ctas));
    }
    std::shuffle(shares.begin(), shares.end(), r);
    for (uint64_t s : shares) {
      if (k == 1 && arrivals >> kArrivalBits != launches) return std::puts("a CTA saw another count"), 1;
      arrivals += s;
    }
    launches += k;
    if (arrivals != launches << kArrivalBits) return std::puts("the count is off"), 1;
  }
}
""")
    r = subprocess.run([exe], capture_output=True, text=True, timeout=120)
    assert r.returncode == 0, r.stdout
